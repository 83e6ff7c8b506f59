// Circuit evaluation in log space (Eq. CP, Eq. HMM, Eq. BTree) and the small preparation kernels.
#pragma once
#include <cuda_bf16.h>
#include <math_constants.h>
#include <stdint.h>

#include "mtpc_ptx.cuh"

namespace mtpc {

constexpr int kCircuitWarps = 8;
constexpr unsigned kFull = 0xffffffffu;

// (m, s) represents log-sum-exp = m + log s. Merging tolerates empty operands (m = -inf, s = 0).
__device__ __forceinline__ void lse_merge(float& m, float& s, float m2, float s2) {
  const float mn = fmaxf(m, m2);
  if (mn == -CUDART_INF_F) { m = mn; s = 0.f; return; }
  s = s * __expf(m - mn) + s2 * __expf(m2 - mn);
  m = mn;
}
__device__ __forceinline__ float warp_lse(float val, bool has) {
  float m = has ? val : -CUDART_INF_F;
  float s = has ? 1.f : 0.f;
  if (has && val != val) { m = 0.f; s = val; }   // NaN must survive the max
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(kFull, m, off);
    const float s2 = __shfl_xor_sync(kFull, s, off);
    lse_merge(m, s, m2, s2);
  }
  return m + __logf(s);
}

// Warp-wide maximum; NaN if any lane holds one (so that refused evidence is not lost to the maximum).
__device__ __forceinline__ float warp_max_nan(float x) {
  float m;
  asm volatile("redux.sync.max.NaN.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}
// log-sum-exp of the `count` floats x[0], x[1], ... by one thread. All -inf: -inf; any NaN: NaN.
__device__ __forceinline__ float thread_lse(const float* x, int count) {
  float m = -CUDART_INF_F;
  for (int k = 0; k < count; ++k) m = fmaxf(m, x[k]);
  if (m == -CUDART_INF_F) m = 0.f;
  float s = 0.f;
  for (int k = 0; k < count; ++k) s += __expf(x[k] - m);
  return m + __logf(s);
}

// Eq. (CP): out[w] = LSE_k( log omega[p, k] + sum_i G[w, i, k] ),  p = w / wpp.
__global__ void circuit_cp_kernel(const float* __restrict__ G, const float* __restrict__ logw,
                                  float* __restrict__ out, int W, int wpp, int n, int r, int sum_rows, int raw_mixture) {
  grid_launch_dependents();
  grid_dependency_wait();   // G and log omega come from the kernel before this one
  const int w = blockIdx.x * kCircuitWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= W) return;
  const float* g = G + static_cast<size_t>(w) * n * r;
  const float* lw = logw + static_cast<size_t>(w / wpp) * sum_rows;
  // raw_mixture: logw holds the mixture LOGITS (the few-position draft path with more than 32 components leaves the
  // softmax to its consumers): log omega_k = logit_k - LSE(logits), so LSE(logits) is subtracted from every result.
  float norm = 0.f;
  if (raw_mixture) {
    float m = -CUDART_INF_F, s = 0.f;
    for (int k = lane; k < r; k += 32) lse_merge(m, s, lw[k], 1.f);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float m2 = __shfl_xor_sync(kFull, m, off);
      const float s2 = __shfl_xor_sync(kFull, s, off);
      lse_merge(m, s, m2, s2);
    }
    norm = m + __logf(s);
  }
  float m = -CUDART_INF_F, s = 0.f;
  for (int k = lane; k < r; k += 32) {
    float a = lw[k];
    for (int i = 0; i < n; ++i) a += g[i * r + k];
    if (a != a) { m = 0.f; s = a; continue; }
    lse_merge(m, s, a, 1.f);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(kFull, m, off);
    const float s2 = __shfl_xor_sync(kFull, s, off);
    lse_merge(m, s, m2, s2);
  }
  if (lane == 0) out[w] = m + __logf(s) - norm;
}

// ---------------------------------------------------------------- prefix marginals and slot messages
// The three kernels below write, for every window,
//   prefix[w, i] = log q(x_0..x_i), the joint with the later bytes summed out (Algorithm 3's marginals; may be NULL),
//   msg[w, i, k] = the log-weight of input unit k of slot i given the bytes before it, up to a constant per (w, i) (may
//                  be NULL): log of p(the latent that owns slot i is k, x_0..x_{i-1}). q(x_i | x_<i) is the mixture of the
//                  slot's input units under softmax(msg[w, i, :]), which is all the acceptance stage needs to know of the

// Mixture: msg_i[k] = log omega_k + sum_{j<i} G[j, k], prefix_i = LSE_k msg_{i+1}[k]. One warp per window: lane = component
// for the running sums (all loads of eight slots in flight), then lane = slot for the log-sum-exps, through a padded
// shared tile, so that no slot waits for another one's reduction. Shared memory: cp_prefix_smem_floats per warp.
constexpr int kCpTileSlots = 32;
__host__ __device__ inline int cp_prefix_warp_floats(int n, int r) { return (n < kCpTileSlots ? n : kCpTileSlots) * (r + 1); }
// Slots [i0, i0 + nc) of one window: leaves msg_{i+1}[k] in tile[(i - i0) (r + 1) + k] and, if mw is given, msg_i[k] in
// mw[i r + k]. `first`: the messages of slot i0 (log omega, or the last row of the tile before). Ends with a warp barrier.
__device__ __forceinline__ void cp_prefix_tile(const float* __restrict__ g, const float* first, float* tile,
                                               float* __restrict__ mw, int i0, int nc, int r, int lane) {
  for (int k = lane; k < r; k += 32) {
    float a = first[k];
    for (int c0 = 0; c0 < nc; c0 += 8) {
      float gv[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) gv[q] = c0 + q < nc ? g[(i0 + c0 + q) * r + k] : 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (c0 + q < nc) {
          if (mw != nullptr) mw[(i0 + c0 + q) * r + k] = a;
          a += gv[q];
          tile[(c0 + q) * (r + 1) + k] = a;
        }
    }
  }
  __syncwarp();
}
__global__ void circuit_cp_prefix_kernel(const float* __restrict__ G, const float* __restrict__ logw,
                                         float* __restrict__ out, float* __restrict__ prefix, float* __restrict__ msg, int W,
                                         int wpp, int n, int r, int sum_rows, int raw_mixture) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  grid_dependency_wait();   // G and log omega come from the kernel before this one
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= W) return;
  float* tile = sm + static_cast<size_t>(threadIdx.x >> 5) * cp_prefix_warp_floats(n, r);
  const float* g = G + static_cast<size_t>(w) * n * r;
  const float* lw = logw + static_cast<size_t>(w / wpp) * sum_rows;
  float* mw = msg != nullptr ? msg + static_cast<size_t>(w) * n * r : nullptr;
  float norm = 0.f;                                 // see circuit_cp_kernel
  if (raw_mixture) norm = thread_lse(lw, r);
  for (int i0 = 0; i0 < n; i0 += kCpTileSlots) {
    const int nc = min(kCpTileSlots, n - i0);
    cp_prefix_tile(g, i0 == 0 ? lw : tile + (kCpTileSlots - 1) * (r + 1), tile, mw, i0, nc, r, lane);
    if (lane < nc) {
      const float res = thread_lse(tile + lane * (r + 1), r) - norm;
      if (prefix != nullptr) prefix[static_cast<size_t>(w) * n + i0 + lane] = res;
      if (out != nullptr && i0 + lane == n - 1) out[w] = res;
    }
    __syncwarp();
  }
}

// Eq. (BTree), bottom-up over the heap-ordered latent tree. Node j >= 1 has the table
// logOmega_j[a][b] = logw[p, r + (j-1) r^2 + a r + b] (parent's value a, own value b); the deepest internal node
// n/2-1+m multiplies the input units of tokens 2m and 2m+1. prod[j][z] is the product unit under z_j = z.

// Dynamic work distribution for the kernels whose cost per window is large: every warp takes the next window index
// from a counter that the projection before the launch zeroes, so that all SMs stay busy until the last window.
__device__ __forceinline__ int next_window(unsigned* counter, int lane) {
  unsigned w = 0;
  if (lane == 0) w = atomicAdd(counter, 1u);
  return static_cast<int>(__shfl_sync(kFull, w, 0));
}

// ---- asynchronous staging of an r x r table (global -> shared) by one warp, for kernels that stream one set of
// tables per position from HBM: the copy of the next table is in flight while the current one is reduced.
__device__ __forceinline__ void cp_async_16(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_4(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_16(float* dst, const float* src) { cp_async_16(smem_u32(dst), src); }
__device__ __forceinline__ void cp_async_4(float* dst, const float* src) { cp_async_4(smem_u32(dst), src); }
// The calling threads' share (of `threads`) of copying count floats to shared memory, not committed.
__device__ __forceinline__ void fetch_floats(float* dst, const float* src, int count, int threads) {
  if ((count & 3) == 0 && ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
#pragma unroll 1
    for (int e = threadIdx.x * 4; e < count; e += threads * 4) cp_async_16(dst + e, src + e);
  } else {
#pragma unroll 1
    for (int e = threadIdx.x; e < count; e += threads) cp_async_4(dst + e, src + e);
  }
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// Copies `count` floats; 16 bytes per request when both addresses allow it (count, src and dst multiples of 4 floats).
__device__ __forceinline__ void warp_table_load_async(float* dst, const float* __restrict__ src, int count, int lane) {
  const bool vec = (count & 3) == 0 && ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0;
  if (vec) {
    for (int e = lane * 4; e < count; e += 128) cp_async_16(dst + e, src + e);
  } else {
    for (int e = lane; e < count; e += 32) cp_async_4(dst + e, src + e);
  }
  cp_async_commit();
}
// One sum layer seen from the parent: lane z returns LSE_b(tab[z][b] + pc[b]); the child's table, unpadded [z][b], and its
// vector pc are in shared memory. Lane z walks its row starting at column z, so that the 32 lanes hit 32 different banks. R a multiple of 4 (both arrays 16-byte aligned):
// the row and the child's vector are read as float4, rotated by the lane so that a quarter-warp's requests fall in
// different bank groups, and reduced in registers (max, then sum of exponentials).
template <int R>
__device__ __forceinline__ float sum_layer_staged_vec(const float* tab, const float* pc, int lane) {
  if (lane >= R) return 0.f;
  constexpr int Q = R / 4;
  const float4* row4 = reinterpret_cast<const float4*>(tab + lane * R);
  const float4* pc4 = reinterpret_cast<const float4*>(pc);
  float v[R];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = (q + lane) & (Q - 1);
    const float4 a = row4[j];
    const float4 b = pc4[j];
    v[4 * q] = a.x + b.x;
    v[4 * q + 1] = a.y + b.y;
    v[4 * q + 2] = a.z + b.z;
    v[4 * q + 3] = a.w + b.w;
  }
  float m = v[0];
#pragma unroll
  for (int q = 1; q < R; ++q) m = fmaxf(m, v[q]);
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < R; ++q) s += __expf(v[q] - m);
  float res = (m == -CUDART_INF_F) ? -CUDART_INF_F : m + __logf(s);
  if (s != s) res = s;                             // NaN evidence must survive the max
  return res;
}
__device__ __forceinline__ float sum_layer_staged(const float* tab, const float* pc, int lane, int r) {
  switch (r) {
    case 32: return sum_layer_staged_vec<32>(tab, pc, lane);
    case 16: return sum_layer_staged_vec<16>(tab, pc, lane);
    case 8: return sum_layer_staged_vec<8>(tab, pc, lane);
    case 4: return sum_layer_staged_vec<4>(tab, pc, lane);
    default: break;
  }
  if (lane >= r) return 0.f;
  const float* row = tab + lane * r;
  float m = -CUDART_INF_F;
  for (int b = 0; b < r; ++b) m = fmaxf(m, row[b] + pc[b]);
  float s = 0.f;
  for (int b = 0; b < r; ++b) s += __expf(row[b] + pc[b] - m);
  float res = (m == -CUDART_INF_F) ? -CUDART_INF_F : m + __logf(s);
  if (s != s) res = s;
  return res;
}

// Joint log-probability alone. Shared memory per warp: (n-1) * r floats of prod + 2 * r * r floats (two staged tables). r <= 32.
// The n-2 tables of a position (57 KB at n = 16, r = 32) are read exactly once, in the order the bottom-up pass
// needs them, through a two-deep cp.async pipeline: this kernel is bound by that stream from HBM.
__host__ __device__ inline int btree_warp_floats(int n, int r) { return (n - 1) * r + 2 * r * r; }

__global__ void circuit_btree_kernel(const float* __restrict__ G, const float* __restrict__ logw, float* __restrict__ out,
                                     unsigned* work_counter, int W, int wpp, int n, int r, int sum_rows) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  grid_dependency_wait();   // G, log omega and the zeroed work counter come from the kernels before this one
  const int wib = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  float* prod = sm + static_cast<size_t>(wib) * btree_warp_floats(n, r);
  float* tabs = prod + (n - 1) * r;
  const bool has = lane < r;
  const int first_leaf_node = n / 2 - 1;
  const int rr = r * r;
  const int ntab = n - 2;                          // table t belongs to child c(t) of node j(t), deepest parents first
  auto child_of = [&](int t) { return 2 * (first_leaf_node - 1 - (t >> 1)) + 1 + (t & 1); };
  for (int w = next_window(work_counter, lane); w < W; w = next_window(work_counter, lane)) {
    const float* g = G + static_cast<size_t>(w) * n * r;
    const float* lw = logw + static_cast<size_t>(w / wpp) * sum_rows;
    if (ntab > 0) warp_table_load_async(tabs, lw + r + static_cast<size_t>(child_of(0) - 1) * rr, rr, lane);
    for (int j = n - 2; j >= first_leaf_node; --j) {
      const int m = j - first_leaf_node;
      if (has) prod[j * r + lane] = g[(2 * m) * r + lane] + g[(2 * m + 1) * r + lane];
    }
    __syncwarp();
    float acc = 0.f;
    for (int t = 0; t < ntab; ++t) {
      const int c = child_of(t);
      if (t + 1 < ntab) {
        warp_table_load_async(tabs + ((t + 1) & 1) * rr, lw + r + static_cast<size_t>(child_of(t + 1) - 1) * rr, rr, lane);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();                                  // table t is in shared memory for every lane
      acc += sum_layer_staged(tabs + (t & 1) * rr, prod + c * r, lane, r);
      if (t & 1) {                                   // both children of node j done
        if (has) prod[((c - 2) >> 1) * r + lane] = acc;
        acc = 0.f;
      }
      __syncwarp();                                  // the buffer may be overwritten, prod[j] may be read
    }
    const float res = warp_lse(has ? lw[lane] + prod[lane] : 0.f, has);
    if (lane == 0) out[w] = res;
    __syncwarp();                                    // the next window reuses the warp's shared memory
  }
}

// Whether a sum of products of probabilities, each scaled by its maximum, is no divisor for the gradient that came to it. The build keeps
// subnormal numbers, so 32 products of factors rounded at 2^-149 are off by 2^-144 at most: from 2^-118 on nothing of a sum is lost.
// And a quotient above 2^112 (a state that its evidence alone makes likely) could overflow where quotients are added over many windows.
constexpr float kSumFloor = 0x1p-118f;
__device__ __forceinline__ bool sum_lost(float sum, float gradient) {
  return sum < fmaxf(kSumFloor, fabsf(gradient) * 0x1p-112f);           // (NaN is not lost: it goes on through the quotient)
}
// sum_b tab[lane][b] vec[b] and sum_z vec[z] tab[z][lane] over a table [r, r] and a vector [r] in shared memory (16-byte aligned for r >= 4);
// lanes past r return 0. Rows are read as float4 rotated by the lane (see sum_layer_staged_vec).
template <int R>
__device__ __forceinline__ float row_dot_vec(const float* tab, const float* vec, int lane) {
  constexpr int Q = R / 4;
  const float4 *row4 = reinterpret_cast<const float4*>(tab + lane * R), *v4 = reinterpret_cast<const float4*>(vec);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
  for (int q = 0; q < Q; ++q) {
    const int j = (q + lane) & (Q - 1);
    const float4 a = row4[j], v = v4[j];
    s0 = fmaf(a.x, v.x, s0);
    s1 = fmaf(a.y, v.y, s1);
    s2 = fmaf(a.z, v.z, s2);
    s3 = fmaf(a.w, v.w, s3);
  }
  return (s0 + s1) + (s2 + s3);
}
__device__ __forceinline__ float row_dot(const float* tab, const float* vec, int lane, int r) {
  if (lane >= r) return 0.f;
  if (r == 32) return row_dot_vec<32>(tab, vec, lane);
  if (r == 16) return row_dot_vec<16>(tab, vec, lane);
  if (r == 8) return row_dot_vec<8>(tab, vec, lane);
  float s = 0.f;
  for (int b = 0; b < r; ++b) s = fmaf(tab[lane * r + b], vec[b], s);
  return s;
}
template <int R>
__device__ __forceinline__ float col_dot_vec(const float* tab, const float* vec, int lane) {
  const float4* v4 = reinterpret_cast<const float4*>(vec);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
  for (int q = 0; q < R / 4; ++q) {
    const float4 v = v4[q];
    s0 = fmaf(v.x, tab[(4 * q) * R + lane], s0);
    s1 = fmaf(v.y, tab[(4 * q + 1) * R + lane], s1);
    s2 = fmaf(v.z, tab[(4 * q + 2) * R + lane], s2);
    s3 = fmaf(v.w, tab[(4 * q + 3) * R + lane], s3);
  }
  return (s0 + s1) + (s2 + s3);
}
__device__ __forceinline__ float col_dot(const float* tab, const float* vec, int lane, int r) {
  if (lane >= r) return 0.f;
  if (r == 32) return col_dot_vec<32>(tab, vec, lane);
  if (r == 16) return col_dot_vec<16>(tab, vec, lane);
  if (r == 8) return col_dot_vec<8>(tab, vec, lane);
  float s = 0.f;
  for (int z = 0; z < r; ++z) s = fmaf(vec[z], tab[z * r + lane], s);
  return s;
}
// log-sum-exp of one value per lane (lanes without one pass -inf). All lanes return it.
__device__ __forceinline__ float warp_lse_nan(float x) {
  float m = warp_max_nan(x);
  if (m == -CUDART_INF_F) m = 0.f;
  float s = __expf(x - m);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
  return m + __logf(s);
}
// For every lane in `lost` LSE_q(vec_q + tab[lane * own + q * step]), vec_q in lane q < r and tab in global memory; the others keep `x`.
__device__ __noinline__ float warp_relog(unsigned lost, float x, float vec, const float* __restrict__ tab, int own, int step, int lane, int r) {
  auto entry = [&](unsigned left) { return lane < r && left != 0 ? tab[(__ffs(left) - 1) * own + lane * step] : -CUDART_INF_F; };
  float next = entry(lost);
  do {
    const int z = __ffs(lost) - 1;
    lost &= lost - 1;
    const float y = lane < r ? vec + next : -CUDART_INF_F;
    next = entry(lost);
    const float l = warp_lse_nan(y);
    if (lane == z) x = l;
  } while (lost != 0);
  return x;
}

// Binary tree: every prefix marginal and slot message from one upward and one downward sweep. With
//   S[c][z] = LSE_b(logOmega_c[z][b] + prod[c][b])  the subtree of node c under its parent's value z (all its tokens seen), and
//   D[c][b] = log p(z_c = b, every token left of c's subtree),
// D[root] = log omega_root, D[left child][b] = LSE_z(D[j][z] + logOmega[z][b]), D[right child][b] = LSE_z(D[j][z] + S[left
// sibling][z] + logOmega[z][b]); at the node that owns the tokens 2m and 2m+1: msg_{2m} = D, msg_{2m+1} = D + G[2m], and the
// prefix marginals are their log-sum-exps with the token's own evidence added. S is only needed inside left subtrees.
// That is 2 (n - 2) table passes at most for all n prefixes; re-evaluating each prefix's path to the root took n log n.
// One CTA per window, a warp per node of a level (2 log2 n - 2 levels one after the other instead of 2 (n - 2) tables): the
// position's tables are fetched into shared memory in one go, so a decode-sized call (fewer windows than SMs) waits for one
// memory round trip, and a batch has several windows' tables in flight per SM. tables_in_smem == 0 (they do not fit: n = 64 at
// r = 32): each warp stages the table it needs. A CTA takes a contiguous run of windows and keeps the tables while the
// position stays the same. Measured against one warp per window and a path per prefix: 4096 windows at n = 16, r = 32:
// 256 -> 148 us; 108 windows at n = 8: 36 -> 6 us.
// In shared memory the tables are probabilities, exponentiated once on their way there, so that a step of either sweep is one warp
// maximum, r multiply-adds per lane and one logarithm (r exponentials of sums, a maximum over them and their sum before). A value whose
// sum falls below kSumFloor takes the step once more with logarithms, the warp working on its row or column of the log tables in global
// memory. The logarithm is the full-precision one: the fast one's error is relative away from 1, and these sums of products of
// probabilities lie well below it where a log-sum-exp's lies above, so that log-marginals were off by up to 1.4 times as much as from log tables (rms at
// 300 windows of n = 16, r = 32: 1.65e-6 from log tables, 2.28e-6 with the fast logarithm, 1.58e-6 so; 0.5 % of the prefix call).
// (4096 windows at n = 16, r = 32, inside a draft: 102 -> 96 us, latency of a window's levels; 27 positions of 4 windows at n = 8:
// 8.7 -> 5.8.) Shared memory: btree_prefix_smem_floats.
// One window of a tree sweep, shared by a CTA. vr: pitch of the [r] vectors (r rounded up to 4 floats).
template <int R>                                   // r, where the kernel is built for it (0: any)
struct TreeSweep {
  int n, r, vr, owners, first_leaf_node, depth;    // depth: the owners' level; level L holds the nodes 2^L - 1 .. 2^(L+1) - 2
  int wib, lane, warps;
  float* tabs;                                     // the n - 2 tables, or one tile per warp
  float *S, *D, *gs, *vec;                         // [n - 1][vr], [n - 1][vr], [n][vr], this warp's vector [vr]
  const float* lw;                                 // the position's row of log omega
  bool resident;

  __device__ void init(float* sm, int n_, int r_, bool tables_in_smem) {
    n = n_; r = R > 0 ? R : r_; vr = (r + 3) / 4 * 4;
    owners = n / 2; first_leaf_node = owners - 1; depth = 31 - __clz(owners);
    wib = threadIdx.x >> 5; lane = threadIdx.x & 31; warps = blockDim.x >> 5;
    resident = tables_in_smem;
    tabs = sm;
    S = sm + ((tables_in_smem ? (n - 2) : warps) * r * r + 3) / 4 * 4;
    D = S + (n - 1) * vr;
    gs = D + (n - 1) * vr;
    vec = gs + n * vr + wib * vr;
  }
  __device__ float* after() const { return gs + (n + warps) * vr; }   // the shared memory past the sweep's own
  __device__ const float* log_table(int c) const { return lw + r + static_cast<size_t>(c - 1) * r * r; }
  // Copies `count` log-probabilities to shared memory, by `threads` threads of which this is the `thread`th, ..
  __device__ static bool whole_vectors(const float* src, int count) { return (count & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0; }
  __device__ static void fetch_table(float* dst, const float* __restrict__ src, int count, int thread, int threads) {
    if (whole_vectors(src, count)) {
      for (int e = thread * 4; e < count; e += threads * 4) cp_async_16(dst + e, src + e);
    } else {
      for (int e = thread; e < count; e += threads) cp_async_4(dst + e, src + e);
    }
    cp_async_commit();
  }
  // .. and, once they are there, makes probabilities of those that the thread itself has copied.
  __device__ static void exponentiate(float* dst, const float* src, int count, int thread, int threads) {
    cp_async_wait<0>();
    if (whole_vectors(src, count)) {
#pragma unroll 2
      for (int e = thread * 4; e < count; e += threads * 4) {
        const float4 x = *reinterpret_cast<const float4*>(dst + e);
        *reinterpret_cast<float4*>(dst + e) = make_float4(__expf(x.x), __expf(x.y), __expf(x.z), __expf(x.w));
      }
    } else {
      for (int e = thread; e < count; e += threads) dst[e] = __expf(dst[e]);
    }
  }
  // Start of window w: the position's tables (unless they are still there), its evidence, log omega of the root.
  __device__ void load(const float* __restrict__ g, const float* __restrict__ lw_, bool new_tables) {
    lw = lw_;
    const bool fetch = resident && new_tables;
    if (fetch) fetch_table(tabs, lw + r, (n - 2) * r * r, threadIdx.x, blockDim.x);
    for (int e = threadIdx.x; e < n * r; e += blockDim.x) gs[(e / r) * vr + e % r] = g[e];
    if (threadIdx.x < r) D[threadIdx.x] = lw[threadIdx.x];
    if (fetch) exponentiate(tabs, lw + r, (n - 2) * r * r, threadIdx.x, blockDim.x);
    __syncthreads();
  }
  __device__ const float* table_of(int c) const {  // node c's probabilities; not resident: staged into the warp's own tile
    if (resident) return tabs + (c - 1) * r * r;
    fetch_table(tabs + wib * r * r, log_table(c), r * r, lane, 32);
    exponentiate(tabs + wib * r * r, log_table(c), r * r, lane, 32);
    __syncwarp();
    return tabs + wib * r * r;
  }
  __device__ float prod_of(int c) const {          // lane's entry of the product unit of node c (its subtree given z_c = lane)
    return c >= first_leaf_node ? gs[2 * (c - first_leaf_node) * vr + lane] + gs[(2 * (c - first_leaf_node) + 1) * vr + lane]
                                : S[(2 * c + 1) * vr + lane] + S[(2 * c + 2) * vr + lane];
  }
  __device__ float in_of(int c) const {            // what comes down to node c's table, per parent value
    return D[((c - 1) >> 1) * vr + lane] + ((c & 1) ? 0.f : S[(c - 1) * vr + lane]);
  }
  // exp(x - m) per lane, m the warp's maximum of x (0 if there is none); lanes past r: 0.
  __device__ float scaled(float x, float& m) const {
    if (lane >= r) x = -CUDART_INF_F;
    m = warp_max_nan(x);
    if (m == -CUDART_INF_F) m = 0.f;
    return __expf(x - m);
  }
  __device__ void up() {                           // S of every node that is not on the right edge
    for (int L = depth; L >= 1; --L) {
      for (int c = (1 << L) - 1 + wib; c < (2 << L) - 2; c += warps) {
        const float prod = lane < r ? prod_of(c) : 0.f;
        float m;
        const float e = scaled(prod, m);
        if (lane < r) vec[lane] = e;
        __syncwarp();
        const float q = row_dot(table_of(c), vec, lane, r);
        float sc = m + logf(q);
        const unsigned lost = __ballot_sync(kFull, lane < r && q < kSumFloor);
        if (lost != 0) sc = warp_relog(lost, sc, prod, log_table(c), r, 1, lane, r);
        if (lane < r) S[c * vr + lane] = sc;
        __syncwarp();
      }
      __syncthreads();
    }
  }
  __device__ void down() {                         // D of every node
    for (int L = 1; L <= depth; ++L) {
      for (int c = (1 << L) - 1 + wib; c <= (2 << L) - 2; c += warps) {
        const float in = lane < r ? in_of(c) : 0.f;
        float m;
        const float u = scaled(in, m);
        if (lane < r) vec[lane] = u;
        __syncwarp();
        const float q = col_dot(table_of(c), vec, lane, r);
        float dc = m + logf(q);
        const unsigned lost = __ballot_sync(kFull, lane < r && q < kSumFloor);
        if (lost != 0) dc = warp_relog(lost, dc, in, log_table(c), 1, r, lane, r);
        if (lane < r) D[c * vr + lane] = dc;
        __syncwarp();
      }
      __syncthreads();
    }
  }
};
__host__ __device__ inline size_t btree_prefix_smem_floats(int n, int r, int warps, bool tables_in_smem) {
  const size_t rr = static_cast<size_t>(r) * r, vr = (static_cast<size_t>(r) + 3) / 4 * 4;
  return ((tables_in_smem ? (n - 2) * rr : warps * rr) + 3) / 4 * 4 + (2 * static_cast<size_t>(n - 1) + n + warps) * vr;
}
template <int R>
__global__ void __launch_bounds__(256, 3) circuit_btree_prefix_kernel(const float* __restrict__ G, const float* __restrict__ logw,
                                                                   float* __restrict__ out, float* __restrict__ prefix,
                                                                   float* __restrict__ msg, int W, int wpp, int n, int r_,
                                                                   int sum_rows, int tables_in_smem) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  grid_dependency_wait();   // G and log omega come from the kernels before this one
  const int r = R > 0 ? R : r_;
  TreeSweep<R> t;
  t.init(sm, n, r, tables_in_smem != 0);
  const int w0 = static_cast<int>(static_cast<long long>(blockIdx.x) * W / gridDim.x);
  const int w1 = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * W / gridDim.x);
  int last_pos = -1;
  for (int w = w0; w < w1; ++w) {
    const int pos = w / wpp;
    t.load(G + static_cast<size_t>(w) * n * r, logw + static_cast<size_t>(pos) * sum_rows, pos != last_pos);
    last_pos = pos;
    t.up();
    t.down();
    for (int m = t.wib; m < t.owners; m += t.warps) {    // the tokens 2m and 2m + 1
      const bool has = t.lane < r;
      const float d = has ? t.D[(t.first_leaf_node + m) * t.vr + t.lane] : -CUDART_INF_F;
      const float d1 = has ? d + t.gs[2 * m * t.vr + t.lane] : -CUDART_INF_F;
      const float d2 = has ? d1 + t.gs[(2 * m + 1) * t.vr + t.lane] : -CUDART_INF_F;
      if (msg != nullptr && has) {
        float* mw = msg + (static_cast<size_t>(w) * n + 2 * m) * r + t.lane;
        mw[0] = d;
        mw[r] = d1;
      }
      const float p0 = warp_lse_nan(d1), p1 = warp_lse_nan(d2);
      if (t.lane == 0) {
        if (prefix != nullptr) {
          prefix[static_cast<size_t>(w) * n + 2 * m] = p0;
          prefix[static_cast<size_t>(w) * n + 2 * m + 1] = p1;
        }
        if (out != nullptr && m == t.owners - 1) out[w] = p1;
      }
    }
    __syncthreads();                               // shared memory is reused by the next window
  }
}

// Lanes of a warp that runs an HMM recursion over r <= 32 states (r a power of two): lane = (part, state); with r < 32 the
// rows of a transition table are shared out over min(32 / r, r) parts.
struct HmmLanes {
  int k, part, parts, rows;
  bool active;
};
__device__ __forceinline__ HmmLanes hmm_lanes(int r, int lane) {
  HmmLanes l;
  l.parts = min(32 / r, r);
  l.rows = r / l.parts;
  l.k = lane & (r - 1);
  l.part = lane / r;
  l.active = lane < r * l.parts;
  return l;
}
// One step of the forward recursion: LSE_a(alpha[a] + logA[a][k]) = m + log sum_a exp(alpha[a] - m) A[a][k] for lane's state k
// (every part returns it). alpha: per active lane, -inf elsewhere; NaN in any of them reaches every state. A [r, r] in shared
// memory holds probabilities (LOG_TABLE: their logarithms); ev: 32 floats of the warp's shared memory, not reused before the
// warp's next synchronisation. Every kernel that runs the recursion takes this step, so they return the same bits.
// hmm_forward_sum returns the sum and m.
template <bool LOG_TABLE>
__device__ __forceinline__ float hmm_forward_sum(float alpha, float* ev, const float* A, const HmmLanes& l, int r, float& m) {
  m = warp_max_nan(alpha);
  if (m == -CUDART_INF_F) m = 0.f;
  if (l.part == 0) ev[l.k] = __expf(alpha - m);
  __syncwarp();
  auto entry = [&](float a) { return LOG_TABLE ? __expf(a) : a; };
  const float* col = A + l.part * l.rows * r + l.k;
  const float* ep = ev + l.part * l.rows;
  float s = 0.f;
  if (l.rows == 32) {                                    // r = 32: four chains, the vector read four values at a time
    const float4* e4 = reinterpret_cast<const float4*>(ep);
    float s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const float4 e = e4[a];
      s = fmaf(e.x, entry(col[(4 * a) * 32]), s);
      s1 = fmaf(e.y, entry(col[(4 * a + 1) * 32]), s1);
      s2 = fmaf(e.z, entry(col[(4 * a + 2) * 32]), s2);
      s3 = fmaf(e.w, entry(col[(4 * a + 3) * 32]), s3);
    }
    s = (s + s1) + (s2 + s3);
  } else if (l.active) {
#pragma unroll 4
    for (int a = 0; a < l.rows; ++a) s = fmaf(ep[a], entry(col[a * r]), s);
  }
  for (int off = r; off < r * l.parts; off <<= 1) s += __shfl_xor_sync(kFull, s, off);
  return s;
}
template <bool LOG_TABLE>
__device__ __forceinline__ float hmm_forward_step(float alpha, float* ev, const float* A, const HmmLanes& l, int r) {
  float m;
  const float s = hmm_forward_sum<LOG_TABLE>(alpha, ev, A, l, r, m);
  return m + __logf(s);
}

// Eq. (HMM), forward recursion over the window: with msg_0 = log pi and alpha_i[k] = msg_i[k] + G[i,k],
//   msg_i[k] = LSE_a(alpha_{i-1}[a] + logA_i[a][k]) = m + log sum_a exp(alpha_{i-1}[a] - m) A_i[a][k],  m = max_a alpha_{i-1}[a],
//   prefix_i = LSE_k alpha_i[k], out = prefix_{n-1}.  r <= 32.
// Position p = w / wpp reads logA_i[a][k] at tables[p * table_stride + (i-1) r^2 + a r + k]: contextual transitions (App. H)
// have table_stride = sum_rows (28 KB per position at n = 8, r = 32, read once: the HBM stream that bounds the call then),
// static ones table_stride = 0.
// A CTA's warps work on windows that share tables. They reach shared memory as probabilities: contextual ones (log-probabilities)
// are exponentiated on their way there by all threads, once per position; of static ones a head keeps the probabilities
// (`probabilities`), and a CTA copies them while it still waits for the kernel before it. So a step of the
// recursion is one warp maximum, 32 multiply-adds per lane and one logarithm, with no exponential of a table entry and no
// memory round trip in it. Tables that do not fit (n = 64 at r = 32) go through in chunks of chunk_tables. The prefix log-sum-exps are taken at the
// end, lane = slot. Measured against one warp per window streaming log tables: 8192 windows at n = 8, r = 32: 42 -> 22 us;
// 128 windows at n = 16: 27 -> 13 us. Shared memory: hmm_circuit_smem_floats.
constexpr int kHmmWarps = 8;                                         // at most: launch_circuit gives a CTA fewer where windows are few
__host__ __device__ inline int hmm_circuit_warp_floats(int n, int r, bool with_prefix) {
  return 64 + (with_prefix ? (n * (r + 1) + 3) / 4 * 4 : 0);          // two vectors of 32, alphas [n][r + 1]
}
__host__ __device__ inline size_t hmm_circuit_smem_floats(int n, int r, bool with_prefix, int chunk_tables, int warps) {
  return (static_cast<size_t>(chunk_tables) * r * r + 3) / 4 * 4 +
         static_cast<size_t>(warps) * hmm_circuit_warp_floats(n, r, with_prefix);
}
__global__ void __launch_bounds__(32 * kHmmWarps, 5) circuit_hmm_kernel(
    const float* __restrict__ G, const float* __restrict__ logw, const float* __restrict__ tables, int table_stride,
    float* __restrict__ out, float* __restrict__ prefix, float* __restrict__ msg, int W, int wpp, int n, int r, int sum_rows,
    int chunk_tables, int probabilities) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  const int warps = blockDim.x >> 5;
  const bool early = probabilities && chunk_tables >= n - 1;           // a static set, complete before the call's first kernel lets this in
  if (early) {
    fetch_floats(sm, tables, (n - 1) * r * r, 32 * warps);
    cp_async_commit();
  }
  grid_dependency_wait();   // G and log omega come from the kernel before this one
  if (early) {
    cp_async_wait<0>();
    __syncthreads();
  }
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rr = r * r;
  float* E = sm;
  float* mine = sm + (chunk_tables * rr + 3) / 4 * 4 + wib * hmm_circuit_warp_floats(n, r, prefix != nullptr);
  float* evec = mine;                                      // [2][32], alternating
  float* alphas = mine + 64;
  const HmmLanes l = hmm_lanes(r, lane);
  const int k = l.k, part = l.part;
  const bool active = l.active;
  // work items: a window a warp; contextual tables: of one position
  const int per_pos = table_stride == 0 ? 0 : (wpp + warps - 1) / warps;
  const int items = table_stride == 0 ? (W + warps - 1) / warps : (W / wpp) * per_pos;
  int loaded_pos = early ? 0 : -1, loaded_first = loaded_pos;          // which tables E holds
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    int pos_tab = 0, w;
    bool valid;
    if (table_stride == 0) {
      w = item * warps + wib;
      valid = w < W;
    } else {
      pos_tab = item / per_pos;
      const int j = (item - pos_tab * per_pos) * warps + wib;
      w = pos_tab * wpp + j;
      valid = j < wpp;
    }
    if (!valid) w = 0;
    const float* g = G + static_cast<size_t>(w) * n * r;
    const float* tb = tables + static_cast<size_t>(pos_tab) * table_stride;
    float* mw = msg != nullptr && valid && part == 0 ? msg + static_cast<size_t>(w) * n * r : nullptr;
    float alpha = -CUDART_INF_F, gi = 0.f;
    // the evidence of the later slots: with prefixes, all of it in one trip to the rows the messages will take, else a step ahead of use
    if (prefix != nullptr && valid)
      for (int e = r + lane; e < n * r; e += 32) cp_async_4(alphas + e + (e >> (31 - __clz(r))), g + e);
    if (active && valid) {
      const float l0 = logw[static_cast<size_t>(w / wpp) * sum_rows + k];
      if (mw != nullptr) mw[k] = l0;
      alpha = l0 + g[k];
      if (n > 1 && prefix == nullptr) gi = g[r + k];
    }
    if (prefix != nullptr) {
      if (active && part == 0) alphas[k] = alpha;
      cp_async_commit();
      cp_async_wait<0>();
      __syncwarp();
    }
    for (int t0 = 0; t0 < n - 1; t0 += chunk_tables) {
      const int nt = min(chunk_tables, n - 1 - t0);
      if (loaded_pos != pos_tab || loaded_first != t0) {
        __syncthreads();                                   // every warp is done with what E held
        const float* src = tb + static_cast<size_t>(t0) * rr;
        const int count = nt * rr;
        if (probabilities) {
          fetch_floats(E, src, count, 32 * warps);
          cp_async_commit();
          cp_async_wait<0>();
        } else if ((count & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
          for (int e = threadIdx.x * 4; e < count; e += 32 * warps * 4) {
            const float4 x = *reinterpret_cast<const float4*>(src + e);
            *reinterpret_cast<float4*>(E + e) = make_float4(__expf(x.x), __expf(x.y), __expf(x.z), __expf(x.w));
          }
        } else {
          for (int e = threadIdx.x; e < count; e += 32 * warps) E[e] = __expf(src[e]);
        }
        __syncthreads();
        loaded_pos = pos_tab;
        loaded_first = t0;
      }
      if (!valid) continue;
      for (int i = t0 + 1; i <= t0 + nt; ++i) {
        const float g_next = (prefix == nullptr && active && i + 1 < n) ? g[(i + 1) * r + k] : 0.f;
        if (prefix != nullptr && active) gi = alphas[i * (r + 1) + k];
        const float c = hmm_forward_step<false>(alpha, evec + (i & 1) * 32, E + (i - 1 - t0) * rr, l, r);
        if (mw != nullptr && active) mw[i * r + k] = c;
        alpha = active ? c + gi : -CUDART_INF_F;
        if (prefix == nullptr) gi = g_next;
        if (prefix != nullptr && active && part == 0) alphas[i * (r + 1) + k] = alpha;
      }
    }
    if (valid) {
      if (prefix != nullptr) {
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
          const float res = thread_lse(alphas + i * (r + 1), r);
          prefix[static_cast<size_t>(w) * n + i] = res;
          if (out != nullptr && i == n - 1) out[w] = res;
        }
        __syncwarp();
      } else if (out != nullptr) {
        const float res = warp_lse_nan(part == 0 ? alpha : -CUDART_INF_F);
        if (lane == 0) out[w] = res;
      }
    }
  }
}

// The same recursion, bit for bit, for many positions with contextual tables and one or two windows each: one warp per window streams
// its log tables, the copy of the next one in flight while this one is reduced. circuit_hmm_kernel gives a position to a CTA, whose
// warps beyond the position's windows only help to exponentiate its tables: the shorter way for as many positions as are resident at once, but
// with several rounds of them the idle warps count. Whole calls of a small head in us, there / here: n = 8, r = 32 at 693 positions 27 / 31, at
// 1500 61 / 55, at 4096 170 / 138; n = 16, r = 32 at 400 43 / 57, at 2200 202 / 151; n = 8, r = 8 at 600 36.0 / 37.4, at 4096 68 / 47.
constexpr int kHmmStreamWarps = 4;
__host__ __device__ inline size_t hmm_stream_warp_floats(int n, int r, bool with_prefix) {
  return 2 * static_cast<size_t>(r) * r + hmm_circuit_warp_floats(n, r, with_prefix);
}
__global__ void __launch_bounds__(32 * kHmmStreamWarps) circuit_hmm_stream_kernel(
    const float* __restrict__ G, const float* __restrict__ logw, const float* __restrict__ tables, int table_stride,
    float* __restrict__ out, float* __restrict__ prefix, float* __restrict__ msg, int W, int wpp, int n, int r, int sum_rows) {
  extern __shared__ __align__(16) float sm[];
  grid_dependency_wait();   // G and log omega come from the kernel before this one
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rr = r * r;
  float* evec = sm + wib * hmm_stream_warp_floats(n, r, prefix != nullptr);      // [2][32], alternating
  float* tabs = evec + 64;                                                       // [2][r, r]
  float* alphas = tabs + 2 * rr;
  const HmmLanes l = hmm_lanes(r, lane);
  const int k = l.k;
  const bool keeps = l.active && l.part == 0;
  for (int w = blockIdx.x * kHmmStreamWarps + wib; w < W; w += gridDim.x * kHmmStreamWarps) {
    const float* g = G + static_cast<size_t>(w) * n * r;
    const float* tb = tables + static_cast<size_t>(w / wpp) * table_stride;
    float* mw = msg != nullptr && keeps ? msg + static_cast<size_t>(w) * n * r : nullptr;
    if (n > 1) warp_table_load_async(tabs, tb, rr, lane);
    float alpha = -CUDART_INF_F, gi = 0.f;
    if (l.active) {
      const float l0 = logw[static_cast<size_t>(w / wpp) * sum_rows + k];
      if (mw != nullptr) mw[k] = l0;
      alpha = l0 + g[k];
      if (n > 1) gi = g[r + k];
    }
    if (prefix != nullptr && keeps) alphas[k] = alpha;
    for (int i = 1; i < n; ++i) {
      const float g_next = (l.active && i + 1 < n) ? g[(i + 1) * r + k] : 0.f;
      if (i + 1 < n) {
        warp_table_load_async(tabs + (i & 1) * rr, tb + static_cast<size_t>(i) * rr, rr, lane);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();                                        // table i is in shared memory for every lane
      const float c = hmm_forward_step<true>(alpha, evec + (i & 1) * 32, tabs + ((i - 1) & 1) * rr, l, r);
      if (mw != nullptr) mw[i * r + k] = c;
      alpha = l.active ? c + gi : -CUDART_INF_F;
      gi = g_next;
      if (prefix != nullptr && keeps) alphas[i * (r + 1) + k] = alpha;
      __syncwarp();                                        // the table's buffer may be overwritten
    }
    if (prefix != nullptr) {
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const float res = thread_lse(alphas + i * (r + 1), r);
        prefix[static_cast<size_t>(w) * n + i] = res;
        if (out != nullptr && i == n - 1) out[w] = res;
      }
      __syncwarp();
    } else if (out != nullptr) {
      const float res = warp_lse_nan(l.part == 0 ? alpha : -CUDART_INF_F);
      if (lane == 0) out[w] = res;
    }
  }
  grid_launch_dependents();                                // (at the end: a waiting GEMM would take the L1)
}

// ---------------------------------------------------------------- training loss (Eq. 6)
// Eq. (6): L_j = -(1/N) sum_i (1/V_ij) sum_t log p(x_{t+j} | x_{<t+j}), L = sum_j gamma^(j-1) L_j, over N sequences of
// L positions with overlapping windows. The conditional of slot j given the context and the window's earlier bytes
// is the difference of consecutive prefix log-marginals; V_ij counts the valid (non-negative) targets of slot j in
// sequence i. Two kernels, both with a fixed reduction order, so the result does not change from run to run.
constexpr int kLossThreads = 1024;
// Both kernels that walk a sequence give thread t the slot t % n and the positions t / n, t / n + kLossThreads / n, ..., so
// that a warp's loads of the [T, n] rows are contiguous; the threads of a slot are then added up in a fixed order. (A thread
// per position and slot after slot read every row n times, 4 bytes in every 4 n: 28 + 30 us at n = 16, 4 sequences of 1024
// positions, against 20 + 10.)
__device__ __forceinline__ int loss_rows_per_step(int n) { return kLossThreads / n; }
// x[q * n + j], q < step, added up over q by the whole CTA into x[j] (halving tree: the order depends on n alone).
template <typename T>
__device__ __forceinline__ void loss_add_rows(T* x, int step, int n) {
  const int q = threadIdx.x / n;
  int half = 1;
  while (2 * half < step) half *= 2;
  for (; half > 0; half >>= 1) {
    __syncthreads();
    if (q < half && q + half < step) x[threadIdx.x] += x[threadIdx.x + half * n];
  }
  __syncthreads();
}

// `beside`: runs beside the kernel ahead of it, the last GEMM of a training call, and ends behind it, so that what follows finds both
// complete. The prefixes have to be complete when this kernel starts, for which some kernel between the circuit and that GEMM lets its
// dependents in only after its own wait or is launched plainly (the list at launch_clusters).
// grid = N. partial[i, j] = (1/V_ij) sum_{t valid} (prefix[t, j] - prefix[t, j-1]), 0 if V_ij = 0.
__global__ void __launch_bounds__(kLossThreads) loss_partial_kernel(const float* __restrict__ prefix,
                                                                    const int* __restrict__ targets,
                                                                    float* __restrict__ partial, int L, int n, int beside) {
  grid_launch_dependents();
  if (!beside) grid_dependency_wait();
  __shared__ float ssum[kLossThreads];
  __shared__ int scnt[kLossThreads];
  const int i = blockIdx.x, step = loss_rows_per_step(n), j = threadIdx.x % n;
  float sum = 0.f;
  int cnt = 0;
  if (threadIdx.x < step * n) {
    for (int t = threadIdx.x / n; t < L; t += step) {
      const size_t row = (static_cast<size_t>(i) * L + t) * n;
      if (targets[row + j] >= 0) {
        sum += prefix[row + j] - (j > 0 ? prefix[row + j - 1] : 0.f);
        cnt += 1;
      }
    }
  }
  ssum[threadIdx.x] = sum;
  scnt[threadIdx.x] = cnt;
  loss_add_rows(ssum, step, n);
  loss_add_rows(scnt, step, n);
  if (threadIdx.x < n) {
    const int c = scnt[threadIdx.x];
    partial[static_cast<size_t>(i) * n + threadIdx.x] = c > 0 ? ssum[threadIdx.x] / static_cast<float>(c) : 0.f;
  }
  if (beside) grid_dependency_wait();
}

// One CTA; warp q reduces the slots q, q + warps, ...: slot_loss[j] = -(1/N) sum_i partial[i, j]; then
// loss = sum_j gamma^j slot_loss[j] (j counted from 0).
__global__ void __launch_bounds__(kLossThreads) loss_final_kernel(const float* __restrict__ partial,
                                                                  float* __restrict__ slot_loss,
                                                                  float* __restrict__ loss, int N, int n, float gamma) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j = warp; j < n; j += kLossThreads / 32) {
    float sum = 0.f;
    for (int i = lane; i < N; i += 32) sum += partial[static_cast<size_t>(i) * n + j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
    if (lane == 0) slot_loss[j] = -sum / static_cast<float>(N);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float tot = 0.f, wgt = 1.f;
    for (int j = 0; j < n; ++j) { tot += wgt * slot_loss[j]; wgt *= gamma; }
    *loss = tot;
  }
}

// Coefficients of the prefix log-marginals in Eq. (6). With c[t, j] = -gamma^j / (N V_ij) for a valid target (i the
// sequence of position t) and 0 otherwise, L = sum_t sum_j c[t, j] (P[t, j] - P[t, j-1]) = sum_t sum_j coeff[t, j] P[t, j]
// with coeff[t, j] = c[t, j] - c[t, j+1] (c[t, n] = 0): the weights of the n backward passes. grid = N, n <= 64.
// It needs nothing of the projection it is launched behind and runs beside it, but ends after it: what follows waits for both. (That
// projection lets it in only after its own wait: whoever read the coefficients of the call before is done.)
__global__ void __launch_bounds__(kLossThreads) loss_coeff_kernel(const int* __restrict__ targets,
                                                                  float* __restrict__ coeff, int L, int n, int N,
                                                                  float gamma) {
  grid_launch_dependents();
  __shared__ int scnt[kLossThreads];
  __shared__ float cj[65];
  const int i = blockIdx.x, step = loss_rows_per_step(n), j = threadIdx.x % n;
  int cnt = 0;
  if (threadIdx.x < step * n)
    for (int t = threadIdx.x / n; t < L; t += step) cnt += targets[(static_cast<size_t>(i) * L + t) * n + j] >= 0;
  scnt[threadIdx.x] = cnt;
  loss_add_rows(scnt, step, n);
  if (threadIdx.x < n) {
    float wgt = 1.f;
    for (int q = 0; q < static_cast<int>(threadIdx.x); ++q) wgt *= gamma;
    const int c = scnt[threadIdx.x];
    cj[threadIdx.x] = c > 0 ? -wgt / (static_cast<float>(N) * static_cast<float>(c)) : 0.f;
  }
  if (threadIdx.x == 0) cj[n] = 0.f;
  __syncthreads();
  for (int t = threadIdx.x / n; t < L && threadIdx.x < step * n; t += step) {
    const size_t row = (static_cast<size_t>(i) * L + t) * n;
    const float here = targets[row + j] >= 0 ? cj[j] : 0.f;
    const float next = (j + 1 < n && targets[row + j + 1] >= 0) ? cj[j + 1] : 0.f;
    coeff[row + j] = here - next;
  }
  grid_dependency_wait();
}

// ---------------------------------------------------------------- preparation
// fp32 -> bf16, eight values per thread and step where count and both addresses allow 16-byte accesses (`vec`), else one.
// (One value per thread took 16.6 us for 2005 x 3072 values, a sixth of the copy bandwidth.)
__global__ void __launch_bounds__(256) f32_to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, size_t count,
                                                          int vec) {
  const size_t first = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (vec && first < count / 8) prefetch_l2(src + 8 * first);    // (256 positions of 4 x 8 x 256, d = 256: a call of 10.8 us now 10.6)
  grid_dependency_wait();
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  if (!vec) {
    for (size_t i = first; i < count; i += stride) dst[i] = __float2bfloat16_rn(src[i]);
    return;
  }
  for (size_t i = first; i < count / 8; i += stride) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(src) + 2 * i), b = __ldcs(reinterpret_cast<const float4*>(src) + 2 * i + 1);
    __nv_bfloat162 o[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w), __floats2bfloat162_rn(b.x, b.y),
                           __floats2bfloat162_rn(b.z, b.w)};
    reinterpret_cast<uint4*>(dst)[i] = *reinterpret_cast<const uint4*>(o);
  }
  grid_launch_dependents();
}

}  // namespace mtpc
