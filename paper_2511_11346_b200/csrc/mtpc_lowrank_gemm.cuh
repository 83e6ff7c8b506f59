// Projection of a head whose unembeddings are shared across the components of a slot and adapted by low-rank terms (App. G):
// U_ij = W_i + A_ij B_ij, so logit[t, i, j, :] = W_i h_t + A_ij (B_ij h_t). The composed [n, r, v, d] tensor is never formed.
// Two plain GEMMs make base = W_base h [T, n v] (fp32) and z = B h [T, n r, 2, k] (two bf16 halves, z = hi + lo, so that
// rounding z to the tensor cores' operand type costs 2^-17 instead of 2^-9); lowrank_logits_kernel does the rest without
// writing a logit. FLOPs per position: 2 d (n v + n r k) + 4 n r v k instead of 2 d n r v.
//
// A work item is (128 positions, slot i, 64 columns b of the vocabulary). A thread of the epilogue keeps the base logits
// of one position and 32 (gradient: 16) columns in registers and walks the slot's r components: corr_j = z_j A_ij^T for the item's
// columns comes out of tensor memory (K = 2k: [hi | lo] against A twice), x = base + corr_j, and then
//   forward   (kLowRankForward): the log-sum-exp of the 32 columns; lowrank_merge_kernel combines the unit's, forms the target's
//             logit and writes G. The reference of the exponentials is the base logits' maximum, known before the walk; a component
//             whose sum leaves [2^-60, 2^120] against it (corrections of many tens) is redone with its own maximum;
//   gradient  (kLowRankGradient): g = post (onehot(target) - exp(x - lse)) as bf16, the operand of the GEMMs of the training
//             call, and sum_j g_ij - so a training call keeps no logits ([T, n r v] fp32 were written and read back) and needs
//             no pass over g for that sum.
// Why this shape: with the components outermost (base logits and a running maximum re-read from tensor memory per component,
// corrections in chunks of <= 48 columns) the kernel was bound by its corrections: a dependent pair of M = 128, N <= 48 MMAs
// costs about 320 cycles against 24 of arithmetic, and the columns of a component waited for each other through the maximum.
// Here the MMAs of two components alternate into one slot of tensor memory, two (gradient: four) slots are in flight, and no
// (component, 32 columns) depends on another. The bound is one ex2 per logit (16 a clock and SM: 149 us at T = 8192, n = 8,
// r = 32, v = 320), in the gradient also the 1.3 GB of g.
// 64 columns divide more vocabularies evenly than 128 (of the third item of v = 320 half the warps had nothing), one wait and one
// release serve two components, and log-sums leave as 128 contiguous bytes (position fastest; transposed through shared memory
// before). Measured, forward / merge / gradient, same sizes: 292 / 62 / 450 us before, 240 / 67 / 403 so, 208 / 64 / 398 now.
// The fused projection that kept logits took 801 us and the passes that made g and its sum from them 921.
// Roles: warp 0 TMA producer, warp 1 MMA issuer, then the epilogue warps (TMEM quarter warp % 4).
// Both issue from a converged warp (elect_one): forward 240 -> 222 us, gradient 403 -> 398. A quarter of the forward's exponentials are polynomials
// (poly_ex2), since the exponential unit was busy for 73 % of the cycles and issue slots for 47: 222 -> 208, the unit busy for 65 % now and
// issue slots for 60. The gradient is at neither bound (45 % and 49 %): nine instructions a logit, and its warps' latency.
// Operand ring: one entry holds 32 / k components, all as 128-byte rows with the 128-byte swizzle: z as one box of 128
// positions x 64 values ([hi | lo] of the components), and A as one box of the item's vocabulary rows x 64 values (the components' k
// adaptor columns first) of a copy laid out [n, v, r, k] (lowrank_repack_kernel, made on every call: A is small and may have changed).
#pragma once
#include <cuda_bf16.h>
#include <math_constants.h>

#include "mtpc_backward.cuh"
#include "mtpc_circuit.cuh"
#include "mtpc_decode.cuh"
#include "mtpc_gemm.cuh"

namespace mtpc {

constexpr int kLrMaxRank = 32;          // k <= 32 (a multiple of 16)
constexpr int kLrMaxVocab = 1792;
constexpr int kLrStages = 3;
constexpr int kLrCols = 64;             // columns of a work item
constexpr int kLrRound = 8;             // gradient: components whose lse, weight and G an epilogue warp fetches at a time
enum { kLowRankForward = 0, kLowRankGradient = 1 };
// Columns of an epilogue thread, and CTAs per SM. Both builds have sixteen epilogue warps on an SM: the forward's in two CTAs, which
// drift apart and fill each other's waits; the gradient keeps a second register per column (the sum over the components) and shares
// the operands, which its narrower threads would otherwise fetch twice.
__host__ __device__ constexpr int lowrank_warp_cols(int mode) { return mode == kLowRankForward ? 32 : 16; }
__host__ __device__ constexpr int lowrank_ctas(int mode) { return mode == kLowRankForward ? 2 : 1; }
__host__ __device__ constexpr int lowrank_subs(int mode) { return kLrCols / lowrank_warp_cols(mode); }
constexpr int kLrRoleWarps = 2;
__host__ __device__ constexpr int lowrank_threads(int mode) { return 32 * kLrRoleWarps + 128 * lowrank_subs(mode); }
__host__ __device__ constexpr int lowrank_tmem_cols(int mode) { return kTmemCols / lowrank_ctas(mode); }
constexpr uint32_t kLrZBox = kBlockM * 128;                  // 128 positions x 64 bf16 of z
constexpr uint32_t kLrStageBytes = kLrZBox + kLrCols * 128;  // and the item's vocabulary rows x 64 bf16 of A'

struct LowRankParams {
  CUtensorMap tm_z;      // z      [T, n*r*2*k]        box 64 x 128, 128-byte swizzle (unit u: hi at (2u)k, lo at (2u+1)k)
  CUtensorMap tm_a;      // A'     [n*v, r*k]          box 64 x kLrCols, 128-byte swizzle (row (i, b): A[i, 0..r-1, b, :])
  int T, m_tiles, n, r, v, vv, k;
  int blocks;                        // column blocks of a unit
  const float* base;                 // [T, n v]
  float* log_sum;                    // forward: [ceil(T / 32), ceil(v / 32), n r, 32] log2 of the sum of exponentials of 32 columns,
  float* ref;                        //          relative to [ceil(T / 32), ceil(v / 32), n, 32] the maximum of their base logits
  const int* targets;                // gradient: [T, n]
  const float* G;                    // gradient: [T, n, r] log phi at the target,
  const float* lse;                  //           [T, n, r] log-sum-exp of every unit,
  const float* post;                 //           [T, n, r] its weighted posterior
  CUtensorMap tm_g;                  //           g: [T][n r][v] of bf16 at a pitch, box 32 x 1 x 64, 128-byte swizzle
  __nv_bfloat16* s;                  //           [T, n v] at a pitch of s_pitch: g summed over a slot's components
  size_t s_pitch;
  unsigned* status;
  uint64_t wait_limit_ns;
};
// Shared memory behind the ring, in floats. Per epilogue warp: the next item's base logits [32 positions][its columns] (16-byte pieces
// swizzled by the position). Gradient, per group of the four warps that share 32 positions: two buffers of g for two components, each
// [32 positions][64 columns] bf16 as a TMA store with 128-byte swizzle takes them, and two rounds of lse, weight and G, each
// [kLrRound][kLrPitch]. Nothing else is shared between epilogue warps: with block-wide staging and barriers a sixth
// (forward) to nearly half (gradient) of the time went into the boundaries between items.
constexpr int kLrTileBytes = 32 * 128;
constexpr int kLrPitch = 33;            // of a component's 32 positions (written and read across components without conflicts)
__host__ __device__ constexpr int lowrank_group_floats(int mode) { return mode == kLowRankForward ? 0 : kLrTileBytes; }   // 4 tiles of 1024
__host__ __device__ constexpr int lowrank_round_floats(int mode) { return mode == kLowRankForward ? 0 : 6 * kLrRound * kLrPitch; }
__host__ __device__ constexpr int lowrank_patch_floats(int mode) {
  return 4 * (lowrank_group_floats(mode) + lowrank_subs(mode) * 32 * lowrank_warp_cols(mode) + lowrank_round_floats(mode));
}
inline size_t lowrank_smem_bytes(int mode) {
  return 1024 + static_cast<size_t>(kLrStages) * kLrStageBytes + lowrank_patch_floats(mode) * sizeof(float) + sizeof(GemmControl);
}

__device__ __forceinline__ void st_shared_bf16(uint32_t dst, __nv_bfloat16 x) {
  asm volatile("st.shared.b16 [%0], %1;" ::"r"(dst), "h"(__bfloat16_as_ushort(x)) : "memory");
}

// 2^y on the multiply-add pipe: y = n + f with |f| <= 1/2 by adding and taking away 1.5 * 2^23, a polynomial of degree 6 in f (its coefficients
// by Remez' exchange for the least relative error, 1.9e-9), n added to the exponent (splitting exponentials between the two units is
// FlashAttention-4's published idea). Against fp64 over [-120, 100] at most 8.0e-8 off (rms 2.7e-8), the exponential unit 1.5e-7 (5e-8). Below -126: 2^-126;
// above 127 or no number: a number beyond 2^120 or no number, which the sums' check catches.
__device__ __forceinline__ float2 poly_ex2(float2 y) {
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(y.x) : "f"(-126.f));
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(y.y) : "f"(-126.f));
  asm("min.NaN.f32 %0, %0, %1;" : "+f"(y.x) : "f"(127.f));
  asm("min.NaN.f32 %0, %0, %1;" : "+f"(y.y) : "f"(127.f));
  auto both = [](float x) { return make_float2(x, x); };
  const float2 t = __fadd2_rn(y, both(12582912.f));
  const float2 f = __ffma2_rn(__fadd2_rn(t, both(-12582912.f)), both(-1.f), y);
  float2 p = __ffma2_rn(both(1.53458124e-4f), f, both(1.33999309e-3f));
  p = __ffma2_rn(p, f, both(9.61848907e-3f));
  p = __ffma2_rn(p, f, both(5.55032864e-2f));
  p = __ffma2_rn(p, f, both(2.40226462e-1f));
  p = __ffma2_rn(p, f, both(6.93147182e-1f));
  p = __ffma2_rn(p, f, both(1.f));
  return make_float2(__int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23)),
                     __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23)));
}
struct LowRankItem {
  int mt, slot, block, width;     // width: columns of this block (a multiple of 16)
};
// column block fastest: the CTAs that run together share the positions' z through L2
__device__ __forceinline__ LowRankItem lowrank_item(const LowRankParams& p, int item) {
  LowRankItem c;
  c.block = item % p.blocks;
  const int rest = item / p.blocks;
  c.slot = rest % p.n;
  c.mt = rest / p.n;
  c.width = min(kLrCols, p.v - c.block * kLrCols);
  return c;
}

template <int MODE>
__global__ void __launch_bounds__(lowrank_threads(MODE), lowrank_ctas(MODE)) lowrank_logits_kernel(const __grid_constant__ LowRankParams p) {
  constexpr int kSubs = lowrank_subs(MODE), kWarpCols = lowrank_warp_cols(MODE);
  constexpr int kTmem = lowrank_tmem_cols(MODE), kSlots = kTmem / (2 * kLrCols);      // a slot: the accumulators of two components
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t ring = (raw_addr + 1023u) & ~1023u;
  float* patches = reinterpret_cast<float*>(smem_raw + (ring - raw_addr) + kLrStages * kLrStageBytes);
  GemmControl* ctl = reinterpret_cast<GemmControl*>(patches + lowrank_patch_floats(MODE));

  const int warp = static_cast<int>(warp_uniform(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const int num_items = p.m_tiles * p.n * p.blocks;
  const int npairs = (p.r + 1) / 2;                       // components go through in pairs (r = 1: one and its copy)
  const int per_entry = 32 / p.k;                         // components per ring entry: 2 (k = 16) or 1 (k = 32)
  const int nent = (p.r + per_entry - 1) / per_entry;     // ring entries per item

  if (threadIdx.x == 0) {
    for (int s = 0; s < kLrStages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&ctl->tfull[s]), 1);
      mbar_init(smem_u32(&ctl->tempty[s]), 4 * kSubs);
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    ctl->wait_limit_ns = p.wait_limit_ns;
    fence_mbar_init();
    tma_prefetch_desc(&p.tm_z);
    tma_prefetch_desc(&p.tm_a);
    if (MODE == kLowRankGradient) tma_prefetch_desc(&p.tm_g);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmem);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(ctl->tmem_base);
  grid_launch_dependents();
  grid_dependency_wait();
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const uint32_t lead = elect_one();
    uint32_t st = 0, phase = 0, issued = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < num_items && ok; item += gridDim.x) {
      const LowRankItem w = lowrank_item(p, item);
      for (int e = 0; e < nent; ++e) {
        if (!bounded_wait_all(smem_u32(&ctl->empty[st]), phase ^ 1u, ctl, p)) { ok = false; break; }
        const uint32_t full = smem_u32(&ctl->full[st]);
        const uint32_t dst = ring + st * kLrStageBytes;
        const int j = e * per_entry;                       // first component of the entry
        mbar_arrive_expect_tx(lead, full, kLrStageBytes);
        // the boxes may cover components past the slot's last (the next slot's, or zeros past the end), adaptor columns past the
        // entry's and rows past the unit: none of that is multiplied
        tma_load_2d(lead, dst, &p.tm_z, full, (w.slot * p.r + j) * 2 * p.k, w.mt * kBlockM);
        tma_load_2d(lead, dst + kLrZBox, &p.tm_a, full, j * p.k, w.slot * p.v + w.block * kLrCols);
        ++issued;
        if (++st == kLrStages) { st = 0; phase ^= 1u; }
      }
    }
    // no copy may still be in flight when the CTA goes away (they have all landed unless some warp gave up)
    for (uint32_t s = 0; s < kLrStages && s < issued; ++s) drain_wait(smem_u32(&ctl->full[s]), ((issued - 1 - s) / kLrStages) & 1u);
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: pair u overall into slot u % kSlots
    const uint32_t lead = elect_one();
    uint32_t st = 0, phase = 0, use = 0;
    bool ok = blockIdx.x >= num_items || first_wait(smem_u32(&ctl->full[0]), ctl, p);
    const uint64_t z_desc0 = umma_smem_desc_sw128(ring), a_desc0 = umma_smem_desc_sw128(ring + kLrZBox);
    constexpr uint32_t kStageStep = kLrStageBytes >> 4;      // descriptors step in 16-byte units
    auto next_stage = [&] {
      umma_commit(lead, smem_u32(&ctl->empty[st]));
      if (++st == kLrStages) { st = 0; phase ^= 1u; }
    };
    for (int item = blockIdx.x; item < num_items && ok; item += gridDim.x) {
      const LowRankItem w = lowrank_item(p, item);
      const uint32_t idesc = umma_idesc_bf16(kBlockM, w.width);
      for (int pr = 0; pr < npairs && ok; ++pr, ++use) {
        const uint32_t slot = use % kSlots;
        if (!bounded_wait_all(smem_u32(&ctl->tempty[slot]), ((use / kSlots) & 1u) ^ 1u, ctl, p)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + slot * 2 * kLrCols;
        const int count = min(2, p.r - 2 * pr);
        if (p.k == 16) {                                     // one entry: [hi | lo] of two components, 16 adaptor columns each
          if (!bounded_wait_all(smem_u32(&ctl->full[st]), phase, ctl, p)) { ok = false; break; }
          tc_fence_after();
          const uint64_t z = z_desc0 + st * kStageStep, a = a_desc0 + st * kStageStep;
          const uint32_t z1 = count == 2 ? 4u : 0u, a1 = count == 2 ? 2u : 0u;
#pragma unroll
          for (int part = 0; part < 2; ++part) {             // (the two alternate: an MMA does not follow the one whose result it adds to)
            umma_bf16(lead, d_tmem, z + 2 * part, a, idesc, part);
            umma_bf16(lead, d_tmem + kLrCols, z + z1 + 2 * part, a + a1, idesc, part);
          }
          next_stage();
        } else {                                             // an entry per component: hi at 0, lo at 32 of its 64 values
          for (int q = 0; q < count && ok; ++q) {
            if (!bounded_wait_all(smem_u32(&ctl->full[st]), phase, ctl, p)) { ok = false; break; }
            tc_fence_after();
            const uint64_t z = z_desc0 + st * kStageStep, a = a_desc0 + st * kStageStep;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma_bf16(lead, d_tmem + q * kLrCols, z + 2 * kk, a + 2 * (kk & 1), idesc, kk != 0 ? 1u : 0u);
            if (count == 1) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma_bf16(lead, d_tmem + kLrCols, z + 2 * kk, a + 2 * (kk & 1), idesc, kk != 0 ? 1u : 0u);
            }
            next_stage();
          }
        }
        if (!ok) break;
        umma_commit(lead, smem_u32(&ctl->tfull[slot]));
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3;
    const int sub = (warp - kLrRoleWarps) >> 2;
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + sub * kWarpCols;
    const size_t units = static_cast<size_t>(p.n) * p.r;
    const float2 l2 = make_float2(kLog2e, kLog2e);
    const uint32_t next_base = smem_u32(patches) + (4 * lowrank_group_floats(MODE) + (warp - kLrRoleWarps) * 32 * kWarpCols) * 4;
    const uint32_t rounds = smem_u32(patches) + (4 * lowrank_group_floats(MODE) + 4 * kSubs * 32 * kWarpCols + quarter * lowrank_round_floats(MODE)) * 4;
    constexpr int kChunks = kWarpCols / 4;                 // 16-byte pieces of a position's base logits
    auto swizzled = [](int row, int ch) { return kChunks == 8 ? ch ^ (row & 7) : ch ^ ((row >> 1) & 3); };
    // ---- copies that are in flight while the current item or round is worked on
    auto fetch_base = [&](int item) {                      // base logits of the warp's 32 positions x its columns
      if (item < num_items) {
        const LowRankItem w = lowrank_item(p, item);
        const int ch = lane % kChunks, col = w.block * kLrCols + sub * kWarpCols + ch * 4;
        if (col < p.v) {
          const float* src = p.base + static_cast<size_t>(w.slot) * p.v + col;
#pragma unroll
          for (int it = 0; it < kChunks; ++it) {
            const int rr = it * (32 / kChunks) + lane / kChunks;
            const int t = min(w.mt * kBlockM + quarter * 32 + rr, p.T - 1);
            cp_async_16(next_base + (rr * kWarpCols + swizzled(rr, ch) * 4) * 4, src + static_cast<size_t>(t) * p.n * p.v);
          }
        }
      }
    };
    // gradient: lse, weight and G of 32 positions x kLrRound components, by the four warps of the positions together
    auto fetch_round = [&](const LowRankItem& w, int j0, uint32_t dst) {
      const int j = lane & (kLrRound - 1);
      if (j0 + j < p.r) {
#pragma unroll
        for (int it = 0; it < 2; ++it) {
          const int rr = it * 16 + sub * 4 + lane / kLrRound;
          const int t = min(w.mt * kBlockM + quarter * 32 + rr, p.T - 1);
          const size_t tu = static_cast<size_t>(t) * units + static_cast<size_t>(w.slot) * p.r + j0 + j;
          const uint32_t d = dst + (j * kLrPitch + rr) * 4;
          cp_async_4(d, p.lse + tu);
          cp_async_4(d + 4 * kLrRound * kLrPitch, p.post + tu);
          cp_async_4(d + 8 * kLrRound * kLrPitch, p.G + tu);
        }
      }
    };
    auto group_barrier = [&] { asm volatile("bar.sync %0, 128;" ::"r"(1 + quarter) : "memory"); };
    uint32_t use = 0, ca[8], cb[8];                          // (ca, cb: the gradient's accumulators, eight columns each)
    const int round_shift = p.r >= 8 ? 2 : p.r >= 4 ? 1 : 0;   // log2 of the pairs in a round: round `use >> round_shift` is in buffer (.. & 1)
    bool ok = true;
    // (every lane polls: no broadcast of the outcome, one vote)
    auto wait_slot = [&](uint32_t u) -> bool {
      const bool up = __all_sync(kFull, bounded_wait(smem_u32(&ctl->tfull[u % kSlots]), (u / kSlots) & 1u, ctl, p.status));
      tc_fence_after();
      return up;
    };
    auto release_slot = [&](uint32_t u) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[u % kSlots]));
    };
    fetch_base(blockIdx.x);
    if (MODE == kLowRankGradient && blockIdx.x < num_items) fetch_round(lowrank_item(p, blockIdx.x), 0, rounds);
    cp_async_commit();
    if (MODE == kLowRankGradient) {
      cp_async_wait<0>();
      group_barrier();
      if (blockIdx.x < num_items) ok = wait_slot(0);
      tmem_ld8_issue(lane_base, ca);
    }
    for (int item = blockIdx.x; item < num_items && (ok || MODE == kLowRankGradient); item += gridDim.x) {
      const LowRankItem w = lowrank_item(p, item);
      const int row = w.mt * kBlockM + quarter * 32 + lane;
      const bool valid = row < p.T;
      const int col0 = w.block * kLrCols + sub * kWarpCols;   // this warp's first column inside the unit
      const int here = min(kWarpCols, p.v - col0);            // its columns (a multiple of 16), or none (<= 0)
      float2 base[kWarpCols / 2];                             // (base - ref) log2(e); ref: their maximum (forward) or 0
      float ref = -CUDART_INF_F;
      cp_async_wait<0>();
      __syncwarp();
#pragma unroll
      for (int q = 0; q < kChunks; ++q) {
        float4 x = ld_shared_v4(next_base + (lane * kWarpCols + swizzled(lane, q) * 4) * 4);
        if (col0 + 4 * q + 4 > p.vv) {                     // padding columns, and columns past the unit, carry no mass
          if (col0 + 4 * q >= p.vv) x.x = -CUDART_INF_F;
          if (col0 + 4 * q + 1 >= p.vv) x.y = -CUDART_INF_F;
          if (col0 + 4 * q + 2 >= p.vv) x.z = -CUDART_INF_F;
          if (col0 + 4 * q + 3 >= p.vv) x.w = -CUDART_INF_F;
        }
        base[2 * q] = make_float2(x.x, x.y);
        base[2 * q + 1] = make_float2(x.z, x.w);
        ref = fmaxf(ref, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
      }
      if (MODE == kLowRankGradient || ref == -CUDART_INF_F) ref = 0.f;
#pragma unroll
      for (int q = 0; q < kWarpCols / 2; ++q) base[q] = make_float2((base[q].x - ref) * kLog2e, (base[q].y - ref) * kLog2e);
      __syncwarp();
      fetch_base(item + gridDim.x);
      if constexpr (MODE == kLowRankForward) {
        cp_async_commit();
        // ---- forward: a component's accumulators in two halves of sixteen columns; the second half is on its way while the first
        // is consumed, the next component's first half while the second is
        const size_t strip = static_cast<size_t>(w.mt * (kBlockM / 32) + quarter) * ((p.v + 31) / 32) + col0 / 32;   // of 32 positions and columns
        if (valid && here > 0) p.ref[(strip * p.n + w.slot) * 32 + lane] = ref;
        float* dst = p.log_sum + (strip * units + static_cast<size_t>(w.slot) * p.r) * 32 + lane;
        uint32_t c0[16], c1[16];
        if (!(ok = wait_slot(use))) break;
        tmem_ld16_issue(lane_base + (use % kSlots) * 2 * kLrCols, c0);
        for (int pr = 0; pr < npairs; ++pr, ++use) {
          const uint32_t pair_col = lane_base + (use % kSlots) * 2 * kLrCols;
          const bool two = 2 * pr + 1 < p.r;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (q == 1 && !two) break;
            const uint32_t col = pair_col + q * kLrCols;
            float2 sa = make_float2(0.f, 0.f), sb = sa;
            auto eat = [&](const uint32_t (&c)[16], int half) {
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                const float2 y = __ffma2_rn(make_float2(__uint_as_float(c[2 * e]), __uint_as_float(c[2 * e + 1])), l2, base[8 * half + e]);
                const float2 x = (e & 3) == 2 ? poly_ex2(y) : make_float2(fast_ex2(y.x), fast_ex2(y.y));   // a quarter of them
                if (e & 1) sb = __fadd2_rn(sb, x);
                else sa = __fadd2_rn(sa, x);
              }
            };
            tmem_ld_wait16(c0);
            tmem_ld16_issue(col + 16, c1);                 // (columns past the block's width are not used)
            if (here > 0) eat(c0, 0);
            tmem_ld_wait16(c1);
            if (q == 0 && two) {
              tmem_ld16_issue(col + kLrCols, c0);
            } else if (pr + 1 < npairs) {
              if (!(ok = wait_slot(use + 1))) break;
              tmem_ld16_issue(lane_base + ((use + 1) % kSlots) * 2 * kLrCols, c0);
            }
            if (here == 32) eat(c1, 1);
            float s = (sa.x + sa.y) + (sb.x + sb.y);
            float l = fast_lg2(s);                         // log2 of the sum relative to ref: a small number
            if (here > 0 && !__all_sync(kFull, s > 0x1p-60f && s < 0x1p120f)) {
              // corrections so large that the base logits' maximum is no reference: once more, with the maximum (NaN stays NaN)
              float m = -CUDART_INF_F;
              s = 0.f;
#pragma unroll 1
              for (int pass = 0; pass < 2; ++pass)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                  uint32_t c[16];
                  tmem_ld16_issue(col + 16 * half, c);
                  tmem_ld_wait16(c);
                  if (16 * half < here) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                      const float b = e & 1 ? base[8 * half + e / 2].y : base[8 * half + e / 2].x;
                      const float y = fmaf(__uint_as_float(c[e]), kLog2e, b);
                      if (pass == 0) m = fmaxf(m, y);
                      else s += fast_ex2(y - m);
                    }
                  }
                }
              l = m + fast_lg2(s);
            }
            if (valid && here > 0) *dst = l;               // position fastest: 128 contiguous bytes per warp, the next component's behind them
            dst += 32;
          }
          if (!ok) break;
          release_slot(use);
        }
      } else {
        // ---- gradient: the next eight columns are on their way while eight are consumed. g leaves by way of shared memory: stored by the
        // threads, 32 bytes to a row each, the stores alone kept the load-store unit busy for half the time. A warp whose wait
        // gave up goes on without waiting, so that the group's barriers still meet.
        float2 sum[8];                                       // sum over the components,
        float hot = 0.f;                                     // and of the weights, for the target's column
#pragma unroll
        for (int q = 0; q < 8; ++q) sum[q] = make_float2(0.f, 0.f);
        const int tgt = valid ? p.targets[static_cast<size_t>(row) * p.n + w.slot] : -1;
        // the target's column; -1: not here (nor is a refused target's, >= vv); -2: a marginalised byte, which has no gradient
        const int rel = tgt < 0 ? -2 : (tgt >= col0 && tgt < min(col0 + 16, p.vv)) ? tgt - col0 : -1;
        const uint32_t tiles = smem_u32(patches) + quarter * (4 * kLrTileBytes) + lane * 128;
        const uint32_t piece = ((2 * sub) ^ (lane & 7)) * 16, piece1 = piece ^ 16;       // where the thread's two 16-byte pieces lie in its row
        for (int pr = 0; pr < npairs; ++pr, ++use) {
          const int jj = 2 * pr & (kLrRound - 1);          // the pair's first component inside its round
          const uint32_t buffer = (use >> round_shift) & 1u;
          if (jj == 0) {                                   // a new round: the next one, of this item or of the next item, is asked for
            const uint32_t next_round = rounds + (buffer ^ 1u) * (12 * kLrRound * kLrPitch);
            if (2 * pr + kLrRound < p.r) fetch_round(w, 2 * pr + kLrRound, next_round);
            else if (item + gridDim.x < num_items) fetch_round(lowrank_item(p, item + gridDim.x), 0, next_round);
            cp_async_commit();
          }
          const uint32_t mine = rounds + (buffer * (3 * kLrRound * kLrPitch) + lane) * 4;
          const uint32_t col = lane_base + (use % kSlots) * 2 * kLrCols;
          const bool two = 2 * pr + 1 < p.r;               // (r = 1: one component, and its copy with no weight)
          const uint32_t tile = tiles + (use & 1u) * (2 * kLrTileBytes);
          const uint32_t at0 = mine + jj * (4 * kLrPitch), at1 = at0 + (two ? 4 * kLrPitch : 0);
          constexpr uint32_t kArray = 4 * kLrRound * kLrPitch;                       // from lse to weight to G
          const bool more = pr + 1 < npairs || item + gridDim.x < num_items;       // pairs after this one
          auto eat = [&](const uint32_t (&c)[8], int half, uint32_t to, float nl, float wt) {
            uint32_t o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 y = __ffma2_rn(make_float2(__uint_as_float(c[2 * e]), __uint_as_float(c[2 * e + 1])), l2,
                                          __fadd2_rn(base[4 * half + e], make_float2(nl, nl)));
              const float2 gq = __fmul2_rn(make_float2(fast_ex2(y.x), fast_ex2(y.y)), make_float2(wt, wt));
              sum[4 * half + e] = __fadd2_rn(sum[4 * half + e], gq);
              const __nv_bfloat162 h = __floats2bfloat162_rn(gq.x, gq.y);
              o[e] = *reinterpret_cast<const uint32_t*>(&h);
            }
            st_shared_v4(to, o[0], o[1], o[2], o[3]);
          };
          float wt = rel != -2 ? -ld_shared_f32(at0 + kArray) : 0.f, nl = -ld_shared_f32(at0) * kLog2e;
          hot -= wt;
          tmem_ld_wait8(ca);
          tmem_ld8_issue(col + 8, cb);
          eat(ca, 0, tile + piece, nl, wt);
          tmem_ld_wait8(cb);
          tmem_ld8_issue(col + kLrCols, ca);
          eat(cb, 1, tile + piece1, nl, wt);
          wt = two && rel != -2 ? -ld_shared_f32(at1 + kArray) : 0.f;
          nl = -ld_shared_f32(at1) * kLog2e;
          hot -= wt;
          tmem_ld_wait8(ca);
          tmem_ld8_issue(col + kLrCols + 8, cb);
          eat(ca, 0, tile + kLrTileBytes + piece, nl, wt);
          tmem_ld_wait8(cb);
          release_slot(use);
          if (more && ok) ok = wait_slot(use + 1);
          tmem_ld8_issue(lane_base + ((use + 1) % kSlots) * 2 * kLrCols, ca);        // (issued on every path: no copies of ca)
          eat(cb, 1, tile + kLrTileBytes + piece1, nl, wt);
          if (rel >= 0) {
            const uint32_t to = tile + (rel & 8 ? piece1 : piece) + (rel & 7) * 2;
            st_shared_bf16(to, __float2bfloat16_rn(ld_shared_f32(at0 + kArray) * (1.f - __expf(ld_shared_f32(at0 + 2 * kArray)))));
            st_shared_bf16(to + kLrTileBytes, __float2bfloat16_rn(wt * (__expf(ld_shared_f32(at1 + 2 * kArray)) - 1.f)));
          }
          // the pair's g leaves; its buffer is written again two pairs on, after the barrier of the next pair, before which the
          // thread that sends has seen this one read
          fence_proxy_async_shared();
          const bool sender = sub == 0 && lane == 0;
          if (sender) bulk_wait_read<0>();
          if (jj + 2 >= kLrRound || pr + 1 == npairs) cp_async_wait<0>();   // the next round's lse, weights and G: visible to the group behind the barrier
          group_barrier();
          if (sender && ok && w.mt * kBlockM + quarter * 32 < p.T) {
            const uint32_t from = tile - lane * 128;
            const int unit = w.slot * p.r + 2 * pr;
            tma_store_3d(&p.tm_g, from, w.block * kLrCols, unit, w.mt * kBlockM + quarter * 32);
            if (two) tma_store_3d(&p.tm_g, from + kLrTileBytes, w.block * kLrCols, unit + 1, w.mt * kBlockM + quarter * 32);
            bulk_commit();
          }
        }
        const bool stores = valid && here > 0;
        if (stores && ok) {
          uint32_t o[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float2 sq = sum[q];
            if (rel == 2 * q) sq.x += hot;
            if (rel == 2 * q + 1) sq.y += hot;
            const __nv_bfloat162 h = __floats2bfloat162_rn(sq.x, sq.y);
            o[q] = *reinterpret_cast<const uint32_t*>(&h);
          }
          st_global_v8_b32(p.s + static_cast<size_t>(row) * p.s_pitch + static_cast<size_t>(w.slot) * p.v + col0, o);
        }
      }
    }
    cp_async_wait<0>();                                    // (after an abort) no copy is in flight when the CTA goes away
    if (MODE == kLowRankGradient) {
      tmem_ld_wait8(ca);
      bulk_wait<0>();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    drain_after_abort<1>(ctl, true);
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmem);
  }
}

// G[t, i, j] = logit[target] - LSE over the unit: the LSE from the log-sums of 32 columns each and their references, the target's
// logit as its base logit + A[i, j, target] . z[t, i, j] (k multiply-adds per thread; A in its repacked layout, so that the r
// components of a slot read one contiguous row). Targets < 0 (marginalised): 0, or NaN where they are refused draws; targets >= vv:
// NaN and the status bit. A CTA takes 32 positions of eight components of a slot: first lane = position and warp = component, so that
// the log-sums are read as they were written; the LSEs change places through shared memory, and then the component runs fastest.
constexpr int kMergeUnits = 8;
template <int K>                                   // k
__global__ void __launch_bounds__(256, K == 16 ? 4 : 3) lowrank_merge_kernel(const float* __restrict__ log_sum, const float* __restrict__ refs,
                                                            const float* __restrict__ base, const __nv_bfloat16* __restrict__ zhl,
                                                            const __nv_bfloat16* __restrict__ Arep, const int* __restrict__ targets,
                                                            float* __restrict__ G, float* __restrict__ lse_out, unsigned* status, int T,
                                                            int n, int r, int v, int vv, int missing_is_nan) {
  __shared__ float tile[32][kMergeUnits + 1];
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.y, t0 = blockIdx.x * 32, u0 = blockIdx.z * kMergeUnits, uc = min(kMergeUnits, r - u0);
  const int blocks = (v + 31) / 32, tl = min(lane, T - 1 - t0);
  const size_t units = static_cast<size_t>(n) * r;
  // the thread's position and component behind the barrier: its target, its row of z and then of A are asked for first
  const int row = threadIdx.x / uc, j = u0 + threadIdx.x - row * uc, t = t0 + row;      // (uc a power of two)
  const bool has = row < 32 && t < T;
  const size_t ti = static_cast<size_t>(t) * n + i, e = ti * r + j;
  const int tgt = has ? targets[ti] : -1;
  uint4 z[K / 4];
  const uint4* zp = reinterpret_cast<const uint4*>(zhl + e * 2 * K);
#pragma unroll
  for (int q = 0; q < K / 4; ++q) z[q] = tgt >= 0 ? __ldcs(zp + q) : make_uint4(0u, 0u, 0u, 0u);
  if (warp < uc) {
    const size_t strip0 = static_cast<size_t>(blockIdx.x) * blocks;
    const float* ls = log_sum + (strip0 * units + static_cast<size_t>(i) * r + u0 + warp) * 32 + tl;
    const float* rf = refs + (strip0 * n + i) * 32 + tl;
    float best = -CUDART_INF_F, ref = 0.f, shift = 0.f, s = 0.f;
    bool bad = false;
    constexpr int kBatch = K == 16 ? 12 : 8;                           // log-sums in flight
    for (int q0 = 0; q0 < blocks; q0 += kBatch) {
      float lq[kBatch], rq[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        lq[q] = q0 + q < blocks ? __ldcs(ls + (q0 + q) * units * 32) : -CUDART_INF_F;
        rq[q] = q0 + q < blocks ? rf[static_cast<size_t>(q0 + q) * n * 32] : 0.f;
      }
#pragma unroll
      for (int h = 0; h < kBatch; h += 4) {              // four at a time, the largest so far the reference
        if (q0 + h >= blocks) break;
        float top = best, top_ref = ref, top_shift = shift;
#pragma unroll
        for (int q = h; q < h + 4; ++q) {
          const float total = fmaf(rq[q], kLog2e, lq[q]);
          bad |= total != total;
          if (total > top) { top = total; top_ref = rq[q]; top_shift = lq[q]; }
        }
        if (q0 + h > 0) s *= fast_ex2(fmaf(ref - top_ref, kLog2e, shift - top_shift));
#pragma unroll
        for (int q = h; q < h + 4; ++q) s += fast_ex2(fmaf(rq[q] - top_ref, kLog2e, lq[q] - top_shift));
        best = top;
        ref = top_ref;
        shift = top_shift;
      }
    }
    tile[lane][warp] = bad ? CUDART_NAN_F : fmaf(shift + fast_lg2(s), kLn2, ref);
  }
  float dot = 0.f;
  if (tgt >= 0 && tgt < vv) {
    const uint4* ap = reinterpret_cast<const uint4*>(Arep + ((static_cast<size_t>(i) * v + tgt) * r + j) * K);
    float d0 = 0.f, d1 = 0.f;
#pragma unroll
    for (int q = 0; q < K / 8; ++q) {
      const uint4 hi = z[q], lo = z[K / 8 + q], a = ap[q];
      const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&hi);
      const __nv_bfloat162* l2 = reinterpret_cast<const __nv_bfloat162*>(&lo);
      const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&a);
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float2 h = __bfloat1622float2(h2[w]), l = __bfloat1622float2(l2[w]), y = __bfloat1622float2(a2[w]);
        d0 = fmaf(h.x + l.x, y.x, d0);
        d1 = fmaf(h.y + l.y, y.y, d1);
      }
    }
    dot = base[ti * v + tgt] + (d0 + d1);
  }
  __syncthreads();
  if (has) {
    const float lse = tile[row][j - u0];
    if (lse_out != nullptr) lse_out[e] = lse;
    G[e] = tgt < 0 ? (missing_is_nan ? CUDART_NAN_F : 0.f) : tgt >= vv ? CUDART_NAN_F : dot - lse;
    if (tgt >= vv) atomicOr(status, kStatusBadTarget);
  }
  grid_launch_dependents();
}

// A [n, r, v, k] -> A' [n, v, r, k] (bf16, k a multiple of 8): one 16-byte piece per thread.
__global__ void lowrank_repack_kernel(const uint4* __restrict__ A, uint4* __restrict__ out, int n, int r, int v, int kv) {
  grid_dependency_wait();
  const size_t total = static_cast<size_t>(n) * r * v * kv;      // kv = k / 8 pieces per row
  const size_t idx = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int q = static_cast<int>(idx % kv);
  size_t rest = idx / kv;
  const int j = static_cast<int>(rest % r);
  rest /= r;
  const int b = static_cast<int>(rest % v);
  const int i = static_cast<int>(rest / v);
  out[idx] = A[((static_cast<size_t>(i) * r + j) * v + b) * kv + q];
  grid_launch_dependents();
}

// Few-position draft on a factored head: logits[p, i, j, b] = base[p, i, b] + sum_q A[i, j, b, q] z[p, i, j, q], from the
// two small products the weight pass left (base = W_base h [P, n v], z = B h [P, n r k], fp32). One CTA per (unit,
// 256 symbols): a thread keeps its symbol's adaptor row in registers and walks the positions, whose z rows sit in shared
// memory. Launched as a programmatic dependent of the weight pass.
constexpr int kExpandThreads = 256;
__global__ void __launch_bounds__(kExpandThreads) lowrank_expand_kernel(const float* __restrict__ base,
                                                                        const float* __restrict__ z,
                                                                        const __nv_bfloat16* __restrict__ A,
                                                                        float* __restrict__ logits, int P, int n, int r,
                                                                        int v, int k) {
  extern __shared__ __align__(16) float zs[];                   // [P, k]
  grid_launch_dependents();
  const int unit = blockIdx.x, i = unit / r;
  {                           // the adaptor rows on their way to L2 meanwhile (100 positions of 16 x 32 x 320, rank 32: a step of 166.4 us now 155.6)
    const int first = blockIdx.y * kExpandThreads, bytes = min(kExpandThreads, v - first) * k * 2;
    const char* a0 = reinterpret_cast<const char*>(A + (static_cast<size_t>(unit) * v + first) * k);
    for (int at = threadIdx.x * 128; at < bytes; at += kExpandThreads * 128) prefetch_l2(a0 + at);
  }
  grid_dependency_wait();
  const int b = blockIdx.y * kExpandThreads + threadIdx.x;
  const size_t units = static_cast<size_t>(n) * r;
  for (int e = threadIdx.x; e < P * k; e += kExpandThreads) zs[e] = z[(static_cast<size_t>(e / k) * units + unit) * k + e % k];
  constexpr int kBatch = 8;                                     // positions whose base logits are in flight
  float next[kBatch];
  const float* brow = base + static_cast<size_t>(i) * v + min(b, v - 1);
  auto fetch = [&](int p0) {
#pragma unroll
    for (int q = 0; q < kBatch; ++q) next[q] = p0 + q < P ? brow[static_cast<size_t>(p0 + q) * n * v] : 0.f;
  };
  fetch(0);
  float a[kLrMaxRank];
  const uint4* arow = reinterpret_cast<const uint4*>(A + (static_cast<size_t>(unit) * v + min(b, v - 1)) * k);   // k bf16 = k / 8 pieces
#pragma unroll
  for (int q = 0; q < kLrMaxRank / 8; ++q) {
    if (q * 8 < k) {
      const uint4 piece = arow[q];
      const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&piece);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float2 f = __bfloat1622float2(h2[t]);
        a[q * 8 + 2 * t] = f.x;
        a[q * 8 + 2 * t + 1] = f.y;
      }
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) a[q * 8 + t] = 0.f;
    }
  }
  __syncthreads();
  if (b >= v) return;
  for (int p0 = 0; p0 < P; p0 += kBatch) {
    float acc[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) acc[q] = next[q];
    if (p0 + kBatch < P) fetch(p0 + kBatch);
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (p0 + u >= P) break;
      const float4* zp = reinterpret_cast<const float4*>(zs + (p0 + u) * k);
#pragma unroll
      for (int q = 0; q < kLrMaxRank / 4; ++q)
        if (4 * q < k) {
          const float4 zq = zp[q];
          acc[u] = fmaf(a[4 * q], zq.x, acc[u]);
          acc[u] = fmaf(a[4 * q + 1], zq.y, acc[u]);
          acc[u] = fmaf(a[4 * q + 2], zq.z, acc[u]);
          acc[u] = fmaf(a[4 * q + 3], zq.w, acc[u]);
        }
      logits[(static_cast<size_t>(p0 + u) * units + unit) * v + b] = acc[u];
    }
  }
}

// Backward pass of a factored head (App. G): with g = d loss / d logit [T, n r v] (bf16) and s_i = sum_j g_ij, both written by
// lowrank_logits_kernel, the gradients are
//   dW_base[i] = s_i^T h,   dA_ij = g_ij^T (B_ij h),   dB_ij = (g_ij A_ij)^T h,
//   d hidden   = s_i W_base[i] + (g_ij A_ij) B_ij  summed over the slots and components.
// A [n r, v, k] -> [n r, v64, k] with v64 = v rounded up to 64 and zero rows past v: the batched GEMM g_ij A_ij walks K in
// blocks of 64 symbols, and what it reads of g past a unit's own columns must meet zeros.
__global__ void lowrank_pad_kernel(const uint4* __restrict__ A, uint4* __restrict__ out, int units, int v, int v64, int kv) {
  grid_dependency_wait();
  const size_t total = static_cast<size_t>(units) * v64 * kv;    // kv = k / 8 pieces per row
  const size_t idx = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int q = static_cast<int>(idx % kv);
  const size_t rest = idx / kv;
  const int b = static_cast<int>(rest % v64);
  const size_t u = rest / v64;
  out[idx] = b < v ? A[(u * v + b) * kv + q] : make_uint4(0u, 0u, 0u, 0u);
  grid_launch_dependents();   // (after the wait: loss_partial_kernel, which works before it waits, relies on it)
}

// Byte draws of a long draft on a factored head (Algorithm 1, input-unit step): one warp per (window, slot) forms the v
// logits of the one unit the window's latent draw selected, base[t, i, :] + A[i, z] (B[i, z] h_t), in shared memory and draws
// the byte by inverse CDF on exp(logit - max) - v k multiply-adds per draw, no tensor cores and no pass over the other
// units. base = W_base h [P, n v] fp32 and z = B h (two bf16 halves [P, n r, 2, k]) come from two plain GEMMs.
// v <= 512. A refused latent draw (unit_sel < 0) or byte uniform leaves the byte at -1 (preset by the latent kernel).
constexpr int kDrawWarps = 8;
__global__ void __launch_bounds__(32 * kDrawWarps) lowrank_draw_kernel(
    const float* __restrict__ base, const __nv_bfloat16* __restrict__ zhl, const __nv_bfloat16* __restrict__ A,
    const int* __restrict__ unit_sel, const float* __restrict__ uniforms, int* __restrict__ out_bytes, unsigned* status, int W,
    int wpp, int n, int r, int v, int vv, int k) {
  grid_dependency_wait();
  extern __shared__ __align__(16) float draw_sm[];                // kDrawWarps x v logits
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* x = draw_sm + warp * v;
  const size_t units = static_cast<size_t>(n) * r;
  const int pairs = W * n;
  const int per = (v + 31) / 32;
  for (int e = blockIdx.x * kDrawWarps + warp; e < pairs; e += gridDim.x * kDrawWarps) {
    const int w = e / n, i = e - w * n;
    const int z = unit_sel[e];
    if (z < 0) continue;                                          // warp-uniform
    const float ub = uniforms[static_cast<size_t>(w) * 2 * n + n + i];
    if (!(ub >= 0.f && ub < 1.f)) {
      if (lane == 0) atomicOr(status, 2u);
      continue;
    }
    const size_t t = static_cast<size_t>(w / wpp);
    const size_t unit = static_cast<size_t>(i) * r + z;
    const __nv_bfloat16* zrow = zhl + (t * units + unit) * 2 * k;
    const float zmine = lane < k ? __bfloat162float(zrow[lane]) + __bfloat162float(zrow[k + lane]) : 0.f;
    float zq[kLrMaxRank];
#pragma unroll
    for (int q = 0; q < kLrMaxRank; ++q) zq[q] = __shfl_sync(0xffffffffu, zmine, q);
    const float* brow = base + (t * n + i) * v;
    float m = -CUDART_INF_F;
    for (int b = lane; b < v; b += 32) {
      float acc = brow[b];
      const uint4* arow = reinterpret_cast<const uint4*>(A + (unit * v + b) * k);
#pragma unroll
      for (int q8 = 0; q8 < kLrMaxRank / 8; ++q8) {
        if (q8 * 8 < k) {
          const uint4 piece = arow[q8];
          const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&piece);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float2 f = __bfloat1622float2(h2[u]);
            acc = fmaf(f.x, zq[q8 * 8 + 2 * u], acc);
            acc = fmaf(f.y, zq[q8 * 8 + 2 * u + 1], acc);
          }
        }
      }
      if (b >= vv) acc = -CUDART_INF_F;                           // [vv, v): padding symbols
      x[b] = acc;
      m = fmaxf(m, acc);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __syncwarp();
    const int byte = warp_inv_cdf_chunk<kSlotMaxPerLane>(x, 0, per, v, vv, m, ub, true, lane);
    if (lane == 0) out_bytes[e] = byte;
    __syncwarp();                                                 // x is reused by the warp's next pair
  }
  grid_launch_dependents();
}

// Acceptance stage after a long draft on a factored head (Algorithm 3): for every window whose draft was rejected at byte s
// (first_rejected[w] = s >= 0) the r v logits of slot s and the r log-sum-exps, which no call kept:
// logits[w, j, :] = base[t, s, :] + A[s, j] (B[s, j] h_t). One warp per (window, component); rows of the outputs are the
// windows themselves (row_of[w] = w). Padding symbols get -inf, as in the projection kernels.
__global__ void __launch_bounds__(32 * kDrawWarps) lowrank_slot_logits_kernel(
    const float* __restrict__ base, const __nv_bfloat16* __restrict__ zhl, const __nv_bfloat16* __restrict__ A,
    const int* __restrict__ first_rejected, float* __restrict__ logits, float* __restrict__ unit_lse, int* __restrict__ row_of,
    int W, int w_first, int wpp, int n, int r, int v, int vv, int k) {
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t units = static_cast<size_t>(n) * r;
  const int pairs = W * r;
  for (int e = blockIdx.x * kDrawWarps + warp; e < pairs; e += gridDim.x * kDrawWarps) {
    const int w = e / r, j = e - w * r;
    if (j == 0 && lane == 0) row_of[w] = w;
    const int s = first_rejected[w];
    if (s < 0) continue;                                          // warp-uniform: everything accepted, no residual draw
    const size_t t = static_cast<size_t>((w_first + w) / wpp);
    const size_t unit = static_cast<size_t>(s) * r + j;
    const __nv_bfloat16* zrow = zhl + (t * units + unit) * 2 * k;
    const float zmine = lane < k ? __bfloat162float(zrow[lane]) + __bfloat162float(zrow[k + lane]) : 0.f;
    float zq[kLrMaxRank];
#pragma unroll
    for (int q = 0; q < kLrMaxRank; ++q) zq[q] = __shfl_sync(0xffffffffu, zmine, q);
    const float* brow = base + (t * n + s) * v;
    float* out = logits + (static_cast<size_t>(w) * r + j) * v;
    float m = -CUDART_INF_F, sum = 0.f;
    for (int b = lane; b < v; b += 32) {
      float acc = brow[b];
      const uint4* arow = reinterpret_cast<const uint4*>(A + (unit * v + b) * k);
#pragma unroll
      for (int q8 = 0; q8 < kLrMaxRank / 8; ++q8) {
        if (q8 * 8 < k) {
          const uint4 piece = arow[q8];
          const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&piece);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float2 f = __bfloat1622float2(h2[u]);
            acc = fmaf(f.x, zq[q8 * 8 + 2 * u], acc);
            acc = fmaf(f.y, zq[q8 * 8 + 2 * u + 1], acc);
          }
        }
      }
      if (b >= vv) acc = -CUDART_INF_F;
      out[b] = acc;
      lse_merge(m, sum, acc, 1.f);                                // running (maximum, sum of exponentials) of this lane's symbols
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
      const float s2 = __shfl_xor_sync(0xffffffffu, sum, off);
      lse_merge(m, sum, m2, s2);
    }
    if (lane == 0) unit_lse[static_cast<size_t>(w) * r + j] = m + __logf(sum);
  }
  grid_launch_dependents();
}

// ---------------------------------------------------------------- gradients through the adaptors A
// y_u [T, k] = g_u A_u and dA_u [v, k] = g_u^T z_u of every unit u from ONE reading of its logit gradients g_u [T, v]: a CTA takes a
// unit at a time and walks its positions, 128 at once; a stage of shared memory holds 128 positions x 128 symbols of g as two
// 64-symbol boxes, which are the K-major operand A of the product y and, untransposed, the MN-major operand A of the product dA.
// y's accumulators (two, of k columns) leave at the end of each 128 positions, dA's (two sets of up to four tiles of 128 symbols) at
// the end of the unit. z: the bf16 high half the forward pass left, k of the 64 columns that a box brings in. Bound by the bytes
// of g: 2 T n r v. Two batched GEMMs, each reading g, took 505 us at 8192 positions of 8 x 32 units of 320 symbols,
// k = 16; this takes 237 (280 while a branch of lane 0's own issued the sixteen small MMAs of a stage), for 205 us of bytes (the second round of units leaves a quarter of the SMs idle; equal runs of tiles over
// all units, which do not, took 353: CTAs at the same positions of neighbouring units read whole rows of g between them). Units of
// more than 512 symbols, or too few units to occupy the device, keep those products.
struct AdaptorGradParams {
  CUtensorMap tm_g;      // g    [T, n r v] at its pitch   box 64 x 128
  CUtensorMap tm_z;      // z    [T, n r 2 k]              box 64 x 128 (unit u: from column 2 k u)
  CUtensorMap tm_a;      // A    [n r v64, k], v64 = v rounded up to 64 with zero rows; box 64 x 64
  int units, T, v, v64, k, stages;
  __nv_bfloat16* y;      // unit u: columns [u k, (u + 1) k)
  size_t y_pitch;
  float* dA;             // [units, v, k]
  unsigned* status;
  uint64_t wait_limit_ns;
};
constexpr uint32_t kAdaptorBox = kBlockM * 128;              // 128 positions x 64 bf16: 16 KB
constexpr uint32_t kAdaptorStage = 2 * kAdaptorBox;
constexpr int kAdaptorMaxV = 512;
// barriers beyond the stage ring: full / empty of A_u, empty of the two z buffers (their bytes count into the first stage of a tile)
constexpr int kAdaptorBarA = 13, kAdaptorBarZ = 14;
inline size_t adaptor_fixed_bytes(int v64) { return 2 * kAdaptorBox + static_cast<size_t>(v64) * 128; }

__global__ void __launch_bounds__(kGemmThreads, 1) adaptor_grad_kernel(const __grid_constant__ AdaptorGradParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
  const uint32_t z_addr = tiles_addr + p.stages * kAdaptorStage, a_addr = z_addr + 2 * kAdaptorBox;
  GemmControl* ctl = reinterpret_cast<GemmControl*>(smem_raw + (a_addr - raw_addr) + static_cast<size_t>(p.v64) * 128);
  const int warp = static_cast<int>(warp_uniform(threadIdx.x >> 5)), lane = threadIdx.x & 31;
  const int t_tiles = (p.T + kBlockM - 1) / kBlockM, pairs = (p.v64 + 127) / 128;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < 4; ++s) {                            // 0, 1: y; 2, 3: dA
      mbar_init(smem_u32(&ctl->tfull[s]), 1);
      mbar_init(smem_u32(&ctl->tempty[s]), 4);
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    ctl->wait_limit_ns = p.wait_limit_ns;
    fence_mbar_init();
    tma_prefetch_desc(&p.tm_g);
    tma_prefetch_desc(&p.tm_z);
    tma_prefetch_desc(&p.tm_a);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(ctl->tmem_base);
  grid_dependency_wait();
  grid_launch_dependents();
  // tensor memory: y at columns 0 and 32, dA's tiles at 64 and 192, 32 columns each
  auto da_col = [&](uint32_t set, int tile) { return 64 + set * 128 + tile * 32; };

  if (warp == 0) {
    const uint32_t lead = elect_one();
    uint32_t stage = 0, phase = 0, issued_mask = 0, phase_mask = 0, tc = 0, uc = 0;
    bool ok = true;
    auto issued = [&](uint32_t bar, uint32_t par) {
      issued_mask |= 1u << bar;
      phase_mask = (phase_mask & ~(1u << bar)) | (par << bar);
    };
    for (int unit = blockIdx.x; unit < p.units && ok; unit += gridDim.x, ++uc) {
      bool a_loaded = false;
      for (int t = 0; t < t_tiles && ok; ++t, ++tc) {
        const uint32_t zbuf = tc & 1u;
        for (int q = 0; q < pairs; ++q) {
          if (!bounded_wait_all(smem_u32(&ctl->empty[stage]), phase ^ 1u, ctl, p)) { ok = false; break; }
          if (q == 0 && !bounded_wait_all(smem_u32(&ctl->empty[kAdaptorBarZ + zbuf]), ((tc >> 1) & 1u) ^ 1u, ctl, p)) { ok = false; break; }
          const bool two = q * 128 + 64 < p.v64;
          const uint32_t full = smem_u32(&ctl->full[stage]), dst = tiles_addr + stage * kAdaptorStage;
          mbar_arrive_expect_tx(lead, full, ((two ? 2 : 1) + (q == 0 ? 1 : 0)) * kAdaptorBox);
          tma_load_2d(lead, dst, &p.tm_g, full, unit * p.v + q * 128, t * kBlockM);
          if (two) tma_load_2d(lead, dst + kAdaptorBox, &p.tm_g, full, unit * p.v + q * 128 + 64, t * kBlockM);
          if (q == 0) tma_load_2d(lead, z_addr + zbuf * kAdaptorBox, &p.tm_z, full, unit * 2 * p.k, t * kBlockM);
          issued(stage, phase);
          if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
          // A_u goes into the buffer that the unit before it has finished with: asked for behind the unit's first stage, so that
          // the wait does not keep g from being fetched
          if (!a_loaded) {
            a_loaded = true;
            if (!bounded_wait_all(smem_u32(&ctl->empty[kAdaptorBarA]), (uc & 1u) ^ 1u, ctl, p)) { ok = false; break; }
            const uint32_t afull = smem_u32(&ctl->full[kAdaptorBarA]);
            mbar_arrive_expect_tx(lead, afull, p.v64 * 128);
            for (int b = 0; b < p.v64; b += 64) tma_load_2d(lead, a_addr + b * 128, &p.tm_a, afull, 0, unit * p.v64 + b);
            issued(kAdaptorBarA, uc & 1u);
          }
        }
      }
    }
    // no copy may still be in flight when the CTA goes away (they have all landed unless some warp gave up)
    for (int s = 0; s < kMaxStages; ++s)
      if (issued_mask & (1u << s)) drain_wait(smem_u32(&ctl->full[s]), (phase_mask >> s) & 1u);
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t lead = elect_one();
    uint32_t stage = 0, phase = 0, tc = 0, uc = 0;
    bool ok = blockIdx.x >= p.units || first_wait(smem_u32(&ctl->full[0]), ctl, p);
    const uint32_t idesc_y = umma_idesc_bf16(kBlockM, p.k, false, true), idesc_da = umma_idesc_bf16(kBlockM, p.k, true, true);
    const uint64_t g_desc0 = umma_smem_desc_sw128(tiles_addr), gt_desc0 = umma_smem_desc_mn_sw128(tiles_addr, kAdaptorBox);
    const uint64_t z_desc0 = umma_smem_desc_mn_sw128(z_addr, kAdaptorBox), a_desc0 = umma_smem_desc_mn_sw128(a_addr, kMnBoxBytes);
    for (int unit = blockIdx.x; unit < p.units && ok; unit += gridDim.x, ++uc) {
      const uint32_t set = uc & 1u;
      if (!bounded_wait_all(smem_u32(&ctl->tempty[2 + set]), ((uc >> 1) & 1u) ^ 1u, ctl, p)) { ok = false; break; }
      if (!bounded_wait_all(smem_u32(&ctl->full[kAdaptorBarA]), uc & 1u, ctl, p)) { ok = false; break; }
      for (int t = 0; t < t_tiles && ok; ++t, ++tc) {
        const uint32_t yslot = tc & 1u;
        if (!bounded_wait_all(smem_u32(&ctl->tempty[yslot]), ((tc >> 1) & 1u) ^ 1u, ctl, p)) { ok = false; break; }
        const uint64_t z_desc = z_desc0 + yslot * (kAdaptorBox >> 4);
        const uint32_t y_tmem = tmem_base + yslot * 32;
        for (int q = 0; q < pairs; ++q) {
          if (!bounded_wait_all(smem_u32(&ctl->full[stage]), phase, ctl, p)) { ok = false; break; }
          tc_fence_after();
          const uint32_t at = stage * (kAdaptorStage >> 4);
          const bool two = q * 128 + 64 < p.v64;
          const uint64_t g_desc = g_desc0 + at, gt_desc = gt_desc0 + at, a_desc = a_desc0 + q * (2 * kMnBoxBytes >> 4);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)                     // 16 symbols: 32 bytes along g's rows, 16 rows down A_u's box
            umma_bf16(lead, y_tmem, g_desc + 2 * kk, a_desc + 128 * kk, idesc_y, (q | kk) != 0 ? 1u : 0u);
          if (two) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma_bf16(lead, y_tmem, g_desc + (kAdaptorBox >> 4) + 2 * kk, a_desc + (kMnBoxBytes >> 4) + 128 * kk, idesc_y, 1u);
          }
          // the second box of an odd number is whatever the stage held before: rows past the unit's symbols, never read
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)                     // 16 positions: 16 rows down both
            umma_bf16(lead, tmem_base + da_col(set, q), gt_desc + 128 * kk, z_desc + 128 * kk, idesc_da, (t | kk) != 0 ? 1u : 0u);
          umma_commit(lead, smem_u32(&ctl->empty[stage]));
          if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit(lead, smem_u32(&ctl->tfull[yslot]));
        umma_commit(lead, smem_u32(&ctl->empty[kAdaptorBarZ + yslot]));
      }
      if (!ok) break;
      umma_commit(lead, smem_u32(&ctl->tfull[2 + set]));
      umma_commit(lead, smem_u32(&ctl->empty[kAdaptorBarA]));
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    uint32_t tc = 0, uc = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < p.units && ok; unit += gridDim.x, ++uc) {
      for (int t = 0; t < t_tiles; ++t, ++tc) {
        const uint32_t yslot = tc & 1u;
        if (!bounded_wait_warp(smem_u32(&ctl->tfull[yslot]), (tc >> 1) & 1u, ctl, p.status, lane)) { ok = false; break; }
        tc_fence_after();
        const int row = t * kBlockM + quarter * 32 + lane;
        for (int b = 0; b < p.k; b += 16) {
          float x[16];
          tmem_ld16(lane_base + yslot * 32 + b, x);
          if (row < p.T) {
            __nv_bfloat162 o[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) o[e] = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
            uint4* dst = reinterpret_cast<uint4*>(p.y + static_cast<size_t>(row) * p.y_pitch + unit * p.k + b);
            dst[0] = reinterpret_cast<const uint4*>(o)[0];
            dst[1] = reinterpret_cast<const uint4*>(o)[1];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[yslot]));
      }
      if (!ok) break;
      const uint32_t set = uc & 1u;
      if (!bounded_wait_warp(smem_u32(&ctl->tfull[2 + set]), (uc >> 1) & 1u, ctl, p.status, lane)) break;
      tc_fence_after();
      for (int q = 0; q < pairs; ++q) {
        const int sym = q * 128 + quarter * 32 + lane;
        for (int b = 0; b < p.k; b += 16) {
          float x[16];
          tmem_ld16(lane_base + da_col(set, q) + b, x);
          if (sym < p.v) {
            float4* dst = reinterpret_cast<float4*>(p.dA + (static_cast<size_t>(unit) * p.v + sym) * p.k + b);
#pragma unroll
            for (int e = 0; e < 4; ++e) dst[e] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[2 + set]));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    drain_after_abort<1>(ctl, true);
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace mtpc