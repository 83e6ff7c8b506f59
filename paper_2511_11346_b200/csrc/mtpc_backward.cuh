// Backward pass of the window log-likelihood (training, Sec. 4.1 / Eq. 6): gradient of
//     L = sum_t weight[t] * log q(x_t | h_t)
// with respect to the hidden states, the emission weights, the sum-unit weights and the static transition logits.
//
// Stages (host side in mtpc_api.cu):
//   1. forward projection kernel, also keeping the emission logits ([T, n r v] fp32, streamed out of the epilogue) and
//      the log-sum-exp of every input unit (lse [T, n, r]);
//   2. circuit backward (this file): one warp per window runs the upward and the downward pass of the circuit and
//      writes post[w, i, k] = weight * d log q / d G[w, i, k] (the posterior of "token i is emitted by unit k") and
//      dsum[w, :] = weight * d log q / d (sum-unit logits), i.e. posterior minus prior of every sum unit, in bf16;
//   3. logit_gradient_kernel (this file): dlogit = post * (onehot(target) - exp(logit - lse)), one streaming pass over
//      the kept logits, written once as bf16 rows;
//   4. plain bf16 GEMMs (plain_gemm_kernel, this file) on those, every operand read where it lies (the tensor cores
//      take either orientation): d hidden = dlogit W + dsum R, dW = dlogit^T h, dR = dsum^T h.
// Only the training calls materialise the logits (fp32, and their bf16 gradient, as the operands of the two weight-sized
// GEMMs); recomputing them on chip instead was measured: a fourth weight-sized contraction against 0.6 ms of streaming.
#pragma once
#include <cuda_bf16.h>

#include "mtpc_circuit.cuh"
#include "mtpc_gemm.cuh"

namespace mtpc {

// Arguments of the circuit backward kernels: those that differentiate sum_w weight[w] log q(window w), and those of the
// training loss of Eq. 6, which is linear in the prefix log-marginals, L = sum_w sum_j coeff[w, j] log p_j: one kernel per
// family gives every prefix (prefix [W, n]) and the whole gradient.
struct CircuitBackwardArgs {
  const float* G;
  const float* logw;
  const int* targets;
  const float* weight;        // [W]
  const float* coeff;         // [W, n] (Eq. 6)
  float* prefix;              // [W, n] (Eq. 6)
  float* out;                 // [W] log q of the window, or NULL
  float* post;                // [W, n, r]
  __nv_bfloat16* dsum;        // [W, dsum_pitch]
  int dsum_pitch;
  int W, n, r, sum_rows;
};

// ---------------------------------------------------------------- circuit backward: mixture (Eq. CP)
// log q = LSE_k a_k, a_k = log omega_k + sum_i G[i, k]:  d log q / d a_k = rho_k = softmax(a)_k for every slot and for
// the mixture weight; through the softmax of the mixture logits: rho_k - omega_k.
__global__ void circuit_cp_backward_kernel(const CircuitBackwardArgs a_) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int w = blockIdx.x * kCircuitWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= a_.W) return;
  const int n = a_.n, r = a_.r;
  const float* g = a_.G + static_cast<size_t>(w) * n * r;
  const float* lw = a_.logw + static_cast<size_t>(w) * a_.sum_rows;
  const float wt = a_.weight[w];
  float a[4];
  float m = -CUDART_INF_F, s = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = lane + 32 * q;
    a[q] = -CUDART_INF_F;
    if (k < r) {
      a[q] = lw[k];
      for (int i = 0; i < n; ++i) a[q] += g[i * r + k];
      if (a[q] != a[q]) { m = 0.f; s = a[q]; }                           // NaN must survive the maximum
      else lse_merge(m, s, a[q], 1.f);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(kFull, m, off);
    const float s2 = __shfl_xor_sync(kFull, s, off);
    lse_merge(m, s, m2, s2);
  }
  const float logq = m + __logf(s);
  if (lane == 0 && a_.out != nullptr) a_.out[w] = logq;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = lane + 32 * q;
    if (k < r) {
      const float rho = __expf(a[q] - logq);
      for (int i = 0; i < n; ++i)
        a_.post[(static_cast<size_t>(w) * n + i) * r + k] = a_.targets[static_cast<size_t>(w) * n + i] >= 0 ? wt * rho : 0.f;
      a_.dsum[static_cast<size_t>(w) * a_.dsum_pitch + k] = __float2bfloat16_rn(wt * (rho - __expf(lw[k])));
    }
  }
}

// Eq. 6 through the mixture: with rho_j = softmax(msg_{j+1}) the posterior after slot j, dL/dG[i, k] = sum_{j >= i} coeff_j
// rho_j[k] and, through the softmax of the mixture logits, dL/dlogit_k = sum_j coeff_j (rho_j[k] - omega_k). One warp per
// window: the running sums and log-sum-exps of circuit_cp_prefix_kernel (the same bits), then one suffix sum over the slots.
// (One launch per prefix length, each reading G up to its slot and adding into fp32 rows, was 8 launches, two memsets and a
// conversion at n = 8: 50 us with their gaps at 2005 positions, prefixes included, against 5.) Shared memory per warp: n (r + 1) + n floats.
__host__ __device__ inline int cp_loss_warp_floats(int n, int r) { return n * (r + 2); }
__global__ void circuit_cp_loss_backward_kernel(const CircuitBackwardArgs a_) {
  grid_launch_dependents();
  grid_dependency_wait();
  extern __shared__ __align__(16) float sm[];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.x * (blockDim.x >> 5) + wib;
  if (w >= a_.W) return;
  const int n = a_.n, r = a_.r;
  float* tile = sm + static_cast<size_t>(wib) * cp_loss_warp_floats(n, r);
  float* lps = tile + n * (r + 1);
  const float* lw = a_.logw + static_cast<size_t>(w) * a_.sum_rows;
  const float* cw = a_.coeff + static_cast<size_t>(w) * n;
  const int* tg = a_.targets + static_cast<size_t>(w) * n;
  cp_prefix_tile(a_.G + static_cast<size_t>(w) * n * r, lw, tile, nullptr, 0, n, r, lane);
  float csum = 0.f;
  for (int i = lane; i < n; i += 32) {
    const float lp = thread_lse(tile + i * (r + 1), r);
    lps[i] = lp;
    a_.prefix[static_cast<size_t>(w) * n + i] = lp;
    csum += cw[i];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) csum += __shfl_xor_sync(kFull, csum, off);
  __syncwarp();
  for (int k = lane; k < r; k += 32) {
    float acc = 0.f;
    for (int i = n - 1; i >= 0; --i) {
      acc = fmaf(cw[i], __expf(tile[i * (r + 1) + k] - lps[i]), acc);
      a_.post[(static_cast<size_t>(w) * n + i) * r + k] = tg[i] >= 0 ? acc : 0.f;
    }
    a_.dsum[static_cast<size_t>(w) * a_.dsum_pitch + k] = __float2bfloat16_rn(acc - csum * __expf(lw[k]));
  }
}

// ---------------------------------------------------------------- gradient of one row of a transition table
// Lane = row (the conditioning value). For every column b: out[b] = wt * (exp(base + row[b] + pc[b]) - exp(row[b]) * gam),
// i.e. pairwise posterior minus conditional probability times the posterior of the conditioning value (the gradient
// with respect to the row's logits). `row` and `pc` are in shared memory; the results go either to a bf16 row in global
// memory (contextual tables: one set per position), or by atomic adds to an fp32 row in shared memory (static tables,
// summed over the windows). R a multiple of 4: float4 reads rotated by the lane (conflict-free), 8-byte stores.
template <int R>
__device__ __forceinline__ void row_grad_vec(const float* row, const float* pc, float base, float gam, float wt, int lane,
                                             __nv_bfloat16* dst, float* acc_row) {
  constexpr int Q = R / 4;
  const float4* row4 = reinterpret_cast<const float4*>(row);
  const float4* pc4 = reinterpret_cast<const float4*>(pc);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = (q + lane) & (Q - 1);
    const float4 a = row4[j];
    const float4 p = pc4[j];
    const float ox = wt * (__expf(base + a.x + p.x) - __expf(a.x) * gam);
    const float oy = wt * (__expf(base + a.y + p.y) - __expf(a.y) * gam);
    const float oz = wt * (__expf(base + a.z + p.z) - __expf(a.z) * gam);
    const float ow = wt * (__expf(base + a.w + p.w) - __expf(a.w) * gam);
    if (acc_row != nullptr) {
      atomicAdd(acc_row + 4 * j, ox);
      atomicAdd(acc_row + 4 * j + 1, oy);
      atomicAdd(acc_row + 4 * j + 2, oz);
      atomicAdd(acc_row + 4 * j + 3, ow);
    } else {
      __nv_bfloat162 lo = __floats2bfloat162_rn(ox, oy);
      __nv_bfloat162 hi = __floats2bfloat162_rn(oz, ow);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(dst + 4 * j) = pk;
    }
  }
}
__device__ __forceinline__ void row_grad(const float* row, const float* pc, float base, float gam, float wt, int lane, int r,
                                         __nv_bfloat16* dst, float* acc_row) {
  switch (r) {
    case 32: row_grad_vec<32>(row, pc, base, gam, wt, lane, dst, acc_row); return;
    case 16: row_grad_vec<16>(row, pc, base, gam, wt, lane, dst, acc_row); return;
    case 8: row_grad_vec<8>(row, pc, base, gam, wt, lane, dst, acc_row); return;
    case 4: row_grad_vec<4>(row, pc, base, gam, wt, lane, dst, acc_row); return;
    default: break;
  }
  for (int q = 0; q < r; ++q) {                       // start at column `lane` (r a power of two): conflict-free
    const int b = (q + lane) & (r - 1);
    const float la = row[b];
    const float o = wt * (__expf(base + la + pc[b]) - __expf(la) * gam);
    if (acc_row != nullptr) atomicAdd(acc_row + b, o);
    else dst[b] = __float2bfloat16_rn(o);
  }
}

// ---------------------------------------------------------------- circuit backward: HMM (Eq. HMM), forward-backward
// Forward messages alpha_i (kept for all steps in shared memory), backward messages
// beta_{i-1}[a] = LSE_b(logA_i[a][b] + G[i][b] + beta_i[b]). Posterior of the state: gamma_i = exp(alpha_i + beta_i - log q)
// = d log q / d G[i, .]; pairwise posterior xi_i[a][b] = exp(alpha_{i-1}[a] + logA_i[a][b] + G[i][b] + beta_i[b] - log q)
// = d log q / d logA_i[a][b]; through the row softmax of the transition logits: xi_i[a][b] - A_i[a][b] gamma_{i-1}[a].
// Tables as in circuit_hmm_kernel (static: stride 0; contextual: one set per position inside log omega).
// Contextual: the transition-logit gradients go to dsum (bf16, one row per position). Static: they are summed over
// the windows into dT [n-1, r, r] (fp32): per CTA in shared memory first, then one atomicAdd per entry and CTA.
// Shared memory: per warp n*r (alpha) + 2*r*r (tables) + 64 floats; static: + (n-1)*r*r floats per CTA.  r <= 32.
__host__ __device__ inline size_t hmm_backward_warp_floats(int n, int r) {
  return static_cast<size_t>(n) * r + 2 * r * r + 64;             // alphas, two tables, two vectors of 32
}
// The kernel of Eq. 6 takes n more floats for the prefixes and a pitch of r + 1 for the alphas, so that a lane per slot reads them
// without bank conflicts - unless without them more warps fit (n = 54 at r = 32, static, fits no other way), then `wide` is false.
__host__ __device__ inline size_t hmm_loss_warp_floats(int n, int r, bool wide) {
  return wide ? (static_cast<size_t>(n) * (r + 2) + 3) / 4 * 4 + 2 * r * r + 64 : hmm_backward_warp_floats(n, r);
}

__global__ void circuit_hmm_backward_kernel(const CircuitBackwardArgs a_, const float* __restrict__ tables,
                                            int table_stride, float* __restrict__ dT, unsigned* work_counter) {
  grid_launch_dependents();
  grid_dependency_wait();
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int n = a_.n, r = a_.r;
  const int rr = r * r;
  const bool is_static = table_stride == 0;
  float* acc = sm;                                                       // static only: [n-1, r, r]
  float* mine = sm + (is_static ? (n - 1) * rr : 0) + static_cast<size_t>(wib) * hmm_backward_warp_floats(n, r);
  float* alphas = mine;                                                  // [n, r]
  float* tabs = alphas + n * r;
  float* cvec = tabs + 2 * rr;
  const bool has = lane < r;
  const HmmLanes l = hmm_lanes(r, lane);
  if (is_static) {
    for (int e = threadIdx.x; e < (n - 1) * rr; e += blockDim.x) acc[e] = 0.f;
    __syncthreads();
  }
  for (int w = next_window(work_counter, lane); w < a_.W; w = next_window(work_counter, lane)) {
    const float* g = a_.G + static_cast<size_t>(w) * n * r;
    const float* lw = a_.logw + static_cast<size_t>(w) * a_.sum_rows;
    const float* tb = tables + static_cast<size_t>(w) * table_stride;
    const float wt = a_.weight[w];
    const size_t prow = static_cast<size_t>(w) * n * r;
    const size_t drow = static_cast<size_t>(w) * a_.dsum_pitch;
    // ---- forward, keeping every alpha_i
    if (n > 1) warp_table_load_async(tabs, tb, rr, lane);
    float alpha = l.active ? lw[l.k] + g[l.k] : -CUDART_INF_F;
    if (has) alphas[lane] = alpha;
    for (int i = 1; i < n; ++i) {
      if (i + 1 < n) {
        warp_table_load_async(tabs + (i & 1) * rr, tb + static_cast<size_t>(i) * rr, rr, lane);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
      const float c = hmm_forward_step<true>(alpha, cvec, tabs + ((i - 1) & 1) * rr, l, r);
      alpha = l.active ? c + g[i * r + l.k] : -CUDART_INF_F;
      if (has) alphas[i * r + lane] = alpha;
      __syncwarp();
    }
    if (!has) alpha = -CUDART_INF_F;                                     // (the other parts' copies)
    const float logq = warp_lse_nan(alpha);
    if (lane == 0 && a_.out != nullptr) a_.out[w] = logq;
    // ---- backward: tables in reverse order; the table of step n - 1 is still in its buffer
    float beta = 0.f;                                                    // beta_{n-1}
    for (int i = n - 1; i >= 1; --i) {
      if (i < n - 1) {
        cp_async_wait<0>();
        __syncwarp();
      }
      if (i - 1 >= 1) warp_table_load_async(tabs + (i & 1) * rr, tb + static_cast<size_t>(i - 2) * rr, rr, lane);
      const float* A = tabs + ((i - 1) & 1) * rr;
      const bool valid = a_.targets[static_cast<size_t>(w) * n + i] >= 0;
      if (has) {
        const float gamma = __expf(alphas[i * r + lane] + beta - logq);
        a_.post[prow + static_cast<size_t>(i) * r + lane] = valid ? wt * gamma : 0.f;
        cvec[lane] = g[i * r + lane] + beta;
      }
      __syncwarp();
      const float beta_prev = sum_layer_staged(A, cvec, lane, r);        // lane a: LSE_b(logA[a][b] + c[b])
      if (has) {
        const float al = alphas[(i - 1) * r + lane];
        const float gam_prev = __expf(al + beta_prev - logq);
        const size_t off = static_cast<size_t>(r) + static_cast<size_t>(i - 1) * rr + lane * r;
        row_grad(A + lane * r, cvec, al - logq, gam_prev, wt, lane, r, is_static ? nullptr : a_.dsum + drow + off,
                 is_static ? acc + static_cast<size_t>(i - 1) * rr + lane * r : nullptr);
      }
      beta = beta_prev;
      __syncwarp();                                                      // cvec and the table buffer are free again
    }
    if (has) {
      const float gamma0 = __expf(alphas[lane] + beta - logq);
      a_.post[prow + lane] = a_.targets[static_cast<size_t>(w) * n] >= 0 ? wt * gamma0 : 0.f;
      a_.dsum[drow + lane] = __float2bfloat16_rn(wt * (gamma0 - __expf(lw[lane])));
    }
    __syncwarp();
  }
  if (is_static) {
    __syncthreads();
    for (int e = threadIdx.x; e < (n - 1) * rr; e += blockDim.x) {
      const float v = acc[e];
      if (v != 0.f) atomicAdd(dT + e, v);
    }
  }
}

// ---------------------------------------------------------------- Eq. 6 through the HMM in one pass
// The training loss is linear in the prefix log-marginals, L = sum_j coeff[w, j] log p_j, and for the HMM
// p_j = sum_z exp(alpha_j[z]) is the forward message of step j summed over the state (later steps integrate to one). One
// forward recursion therefore gives every prefix, and one reverse sweep gives the whole gradient: with
// abar_i[z] = dL / d alpha_i[z] (plain numbers of either sign, bounded by sum_j |coeff_j|),
//   abar_{n-1} = coeff_{n-1} softmax(alpha_{n-1}),
//   prop_{i-1}[a] = sum_b exp(alpha_{i-1}[a] + logA_i[a][b] + G[i][b] - alpha_i[b]) abar_i[b]     (a conditional probability
//   abar_{i-1}[a] = coeff_{i-1} softmax(alpha_{i-1})[a] + prop_{i-1}[a]                             times abar_i[b])
// and dL/dG[i] = abar_i, dL/d logA_i[a][b] = the summand of prop_{i-1}[a]; through the row softmax of the transition
// logits: summand - A_i[a][b] prop_{i-1}[a]; initial unit: abar_0 - omega sum_z abar_0[z]. Same streaming of the tables
// and the same outputs as circuit_hmm_backward_kernel (post fp32, dsum bf16, static dT by atomics), and the prefixes themselves.
template <int R>
__device__ __forceinline__ void row_grad_mult_vec(const float* row, const float* pc, const float* mult, float base, float gam,
                                                  int lane, __nv_bfloat16* dst, float* acc_row) {
  constexpr int Q = R / 4;
  const float4* row4 = reinterpret_cast<const float4*>(row);
  const float4* pc4 = reinterpret_cast<const float4*>(pc);
  const float4* mu4 = reinterpret_cast<const float4*>(mult);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = (q + lane) & (Q - 1);
    const float4 a = row4[j];
    const float4 p = pc4[j];
    const float4 mu = mu4[j];
    const float ox = __expf(base + a.x + p.x) * mu.x - __expf(a.x) * gam;
    const float oy = __expf(base + a.y + p.y) * mu.y - __expf(a.y) * gam;
    const float oz = __expf(base + a.z + p.z) * mu.z - __expf(a.z) * gam;
    const float ow = __expf(base + a.w + p.w) * mu.w - __expf(a.w) * gam;
    if (acc_row != nullptr) {
      atomicAdd(acc_row + 4 * j, ox);
      atomicAdd(acc_row + 4 * j + 1, oy);
      atomicAdd(acc_row + 4 * j + 2, oz);
      atomicAdd(acc_row + 4 * j + 3, ow);
    } else {
      __nv_bfloat162 lo = __floats2bfloat162_rn(ox, oy);
      __nv_bfloat162 hi = __floats2bfloat162_rn(oz, ow);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(dst + 4 * j) = pk;
    }
  }
}
// Lane = row a of the table: out[b] = exp(base + row[b] + pc[b]) mult[b] - exp(row[b]) gam, to a bf16 row in global memory
// or by atomic adds to an fp32 row in shared memory.
__device__ __forceinline__ void row_grad_mult(const float* row, const float* pc, const float* mult, float base, float gam,
                                              int lane, int r, __nv_bfloat16* dst, float* acc_row) {
  switch (r) {
    case 32: row_grad_mult_vec<32>(row, pc, mult, base, gam, lane, dst, acc_row); return;
    case 16: row_grad_mult_vec<16>(row, pc, mult, base, gam, lane, dst, acc_row); return;
    case 8: row_grad_mult_vec<8>(row, pc, mult, base, gam, lane, dst, acc_row); return;
    case 4: row_grad_mult_vec<4>(row, pc, mult, base, gam, lane, dst, acc_row); return;
    default: break;
  }
  for (int q = 0; q < r; ++q) {
    int b = q + lane;                                   // start at column `lane`: fewer bank conflicts
    if (b >= r) b -= r;
    const float la = row[b];
    const float o = __expf(base + la + pc[b]) * mult[b] - __expf(la) * gam;
    if (acc_row != nullptr) atomicAdd(acc_row + b, o);
    else dst[b] = __float2bfloat16_rn(o);
  }
}

__global__ void circuit_hmm_loss_backward_kernel(const CircuitBackwardArgs a_, const float* __restrict__ tables,
                                                 int table_stride, float* __restrict__ dT, unsigned* work_counter, int wide) {
  grid_launch_dependents();
  grid_dependency_wait();
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int n = a_.n, r = a_.r;
  const int rr = r * r;
  const bool is_static = table_stride == 0;
  float* acc = sm;                                                       // static only: [n-1, r, r]
  float* mine = sm + (is_static ? (n - 1) * rr : 0) + static_cast<size_t>(wib) * hmm_loss_warp_floats(n, r, wide != 0);
  float* tabs = mine;
  float* cvec = tabs + 2 * rr;                                           // G[i] - alpha_i (log domain)
  float* dvec = cvec + 32;                                               // abar_i (plain)
  float* alphas = dvec + 32;                                             // [n][pitch]
  const int pitch = wide ? r + 1 : r;
  const bool has = lane < r;
  const HmmLanes l = hmm_lanes(r, lane);
  if (is_static) {
    for (int e = threadIdx.x; e < (n - 1) * rr; e += blockDim.x) acc[e] = 0.f;
    __syncthreads();
  }
  for (int w = next_window(work_counter, lane); w < a_.W; w = next_window(work_counter, lane)) {
    const float* g = a_.G + static_cast<size_t>(w) * n * r;
    const float* lw = a_.logw + static_cast<size_t>(w) * a_.sum_rows;
    const float* tb = tables + static_cast<size_t>(w) * table_stride;
    const float* cw = a_.coeff + static_cast<size_t>(w) * n;
    const int* tg = a_.targets + static_cast<size_t>(w) * n;
    float* lps = wide ? alphas + n * pitch : a_.prefix + static_cast<size_t>(w) * n;   // [n] the prefix log-marginals
    const size_t prow = static_cast<size_t>(w) * n * r;
    const size_t drow = static_cast<size_t>(w) * a_.dsum_pitch;
    // ---- forward, keeping every alpha_i
    if (n > 1) warp_table_load_async(tabs, tb, rr, lane);
    float alpha = l.active ? lw[l.k] + g[l.k] : -CUDART_INF_F;
    if (has) alphas[lane] = alpha;
    for (int i = 1; i < n; ++i) {
      if (i + 1 < n) {
        warp_table_load_async(tabs + (i & 1) * rr, tb + static_cast<size_t>(i) * rr, rr, lane);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
      const float c = hmm_forward_step<true>(alpha, cvec, tabs + ((i - 1) & 1) * rr, l, r);
      alpha = l.active ? c + g[i * r + l.k] : -CUDART_INF_F;
      if (has) alphas[i * pitch + lane] = alpha;
      __syncwarp();
    }
    if (!has) alpha = -CUDART_INF_F;                                     // (the other parts' copies)
    for (int i = lane; i < n; i += 32) {                                 // every prefix, lane = slot (as circuit_hmm_kernel)
      const float lp = thread_lse(alphas + i * pitch, r);
      lps[i] = lp;
      a_.prefix[static_cast<size_t>(w) * n + i] = lp;
    }
    __syncwarp();
    // ---- reverse sweep: tables in reverse order; the table of step n - 1 is still in its buffer
    float abar = has ? cw[n - 1] * __expf(alpha - lps[n - 1]) : 0.f;
    for (int i = n - 1; i >= 1; --i) {
      if (i < n - 1) {
        cp_async_wait<0>();
        __syncwarp();
      }
      if (i - 1 >= 1) warp_table_load_async(tabs + (i & 1) * rr, tb + static_cast<size_t>(i - 2) * rr, rr, lane);
      const float* A = tabs + ((i - 1) & 1) * rr;
      const float al_i = has ? alphas[i * pitch + lane] : -CUDART_INF_F;
      if (has) {
        a_.post[prow + static_cast<size_t>(i) * r + lane] = tg[i] >= 0 ? abar : 0.f;
        cvec[lane] = al_i == -CUDART_INF_F ? -CUDART_INF_F : g[i * r + lane] - al_i;
        dvec[lane] = abar;
      } else {
        cvec[lane] = -CUDART_INF_F;
        dvec[lane] = 0.f;
      }
      __syncwarp();
      const float al = has ? alphas[(i - 1) * pitch + lane] : -CUDART_INF_F;
      float prop = 0.f;
      if (has) {
        const float* row = A + lane * r;
        for (int q = 0; q < r; ++q) {
          int b = q + lane;
          if (b >= r) b -= r;
          prop += __expf(al + row[b] + cvec[b]) * dvec[b];
        }
        const size_t off = static_cast<size_t>(r) + static_cast<size_t>(i - 1) * rr + lane * r;
        row_grad_mult(row, cvec, dvec, al, prop, lane, r, is_static ? nullptr : a_.dsum + drow + off,
                      is_static ? acc + static_cast<size_t>(i - 1) * rr + lane * r : nullptr);
      }
      abar = has ? cw[i - 1] * __expf(al - lps[i - 1]) + prop : 0.f;
      __syncwarp();                                                      // cvec, dvec and the table buffer are free again
    }
    float total = abar;                                                  // sum_z abar_0[z]
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) total += __shfl_xor_sync(kFull, total, off);
    if (has) {
      a_.post[prow + lane] = tg[0] >= 0 ? abar : 0.f;
      a_.dsum[drow + lane] = __float2bfloat16_rn(abar - __expf(lw[lane]) * total);
    }
    __syncwarp();
  }
  if (is_static) {
    __syncthreads();
    for (int e = threadIdx.x; e < (n - 1) * rr; e += blockDim.x) {
      const float v = acc[e];
      if (v != 0.f) atomicAdd(dT + e, v);
    }
  }
}

// The same for static transitions whose probabilities a head keeps: one set of tables for all windows, so nothing is streamed, no
// table entry is exponentiated, and the table gradients are sums of rank-one terms that need no atomics. With u = exp(alpha_{i-1} -
// max), c_i[b] = sum_a u[a] A[a][b] (the forward step's sum) and x_i[b] = abar_i[b] / c_i[b]:
//   prop_{i-1}[a] = u[a] sum_b A[a][b] x_i[b],   dL/d(logit of A_i[a][b]) = A[a][b] (u[a] x_i[b] - prop_{i-1}[a]).
// A batch is one window per warp: each warp runs its window forward and back (32 multiply-adds a lane and step either way) and leaves
// u, x and prop in shared memory; then the steps are dealt to the warps, which add the batch's u x^T - prop into the CTA's running
// sums, eight columns in registers at a time (acc [n-1][b][a]: lane = a, conflict-free). The factor A and the addition into dT come
// once per CTA. A column b that sum_lost finds takes its part of prop and dT with logarithms: an exponential and at most an atomic per lane,
// and no atomic for what is below the normal numbers, which is all that a state hardly ever entered has to give. (Whole steps redone so, by
// a test that any state with a posterior met: a head with one state entered with e^-75 took 2048 us instead of 58.) Forward step and prefixes
// are those of circuit_hmm_kernel, bit for bit.
// 8192 windows of n = 8, r = 32: 202 us by the streaming kernel (five exponentials an entry, 32 shared atomics a lane and step), 52 by this
// one, bound by its instructions and the reads of the tables from shared memory.
// Shared memory: 2 (n-1) r^2 floats, and per warp hmm_static_loss_warp_floats.
constexpr int kHmmStaticWarps = 16;
__host__ __device__ inline size_t hmm_static_loss_warp_floats(int n, int r) {
  return (static_cast<size_t>(n) * r + 3) / 4 * 4 + 64 + (static_cast<size_t>(n) * (2 * r + 1) + 3) / 4 * 4;
}
// What the columns b in `lost` give to the gradient of the lane's alpha (al) and, if it is `mine` to write, to its row of dT. back: per
// state b (in lane b) its evidence less alpha_i[b]; row: the lane's row of the log table. (Inlined it costs its callers' registers: 0.4 %.)
__device__ __noinline__ float hmm_lost_columns(unsigned lost, float al, float back, float abar, const float* __restrict__ row,
                                               float* dT_row, bool mine) {
  float sum = 0.f;
  do {
    const int b = __ffs(lost) - 1;
    lost &= lost - 1;
    const float back_b = __shfl_sync(kFull, back, b), abar_b = __shfl_sync(kFull, abar, b);
    const float e = __expf(al + row[b] + back_b) * abar_b;
    sum += e;
    if (mine && !(fabsf(e) < 0x1p-126f)) atomicAdd(dT_row + b, e);
  } while (lost != 0);
  return sum;
}
__global__ void __launch_bounds__(32 * kHmmStaticWarps, 2) circuit_hmm_static_loss_backward_kernel(
    const CircuitBackwardArgs a_, const float* __restrict__ prob, const float* __restrict__ logA, float* __restrict__ dT) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int n = a_.n, r = a_.r, rr = r * r, tables = (n - 1) * rr;
  float* E = sm;                                                         // [n-1][r, r]
  float* acc = E + (tables + 3) / 4 * 4;                                 // [n-1][b][a]
  float* area = acc + (tables + 3) / 4 * 4;
  const size_t warp_floats = hmm_static_loss_warp_floats(n, r);
  const int off_u = (n * r + 3) / 4 * 4 + 64, off_prop = off_u + n * (r + 1);
  float* xs = area + wib * warp_floats;                                  // [n][r]: c_i, then x_i
  float* ev = xs + (n * r + 3) / 4 * 4;                                  // two vectors of 32
  float* us = xs + off_u;                                                // [n][r + 1]: alpha_i, then u of the step after it
  float* props = xs + off_prop;                                          // [n][r]
  fetch_floats(E, prob, tables, blockDim.x);                             // static tables: complete before the call's first kernel lets this in
  cp_async_commit();
  for (int e = threadIdx.x; e < tables; e += blockDim.x) acc[e] = 0.f;
  grid_dependency_wait();
  cp_async_wait<0>();
  __syncthreads();
  const HmmLanes l = hmm_lanes(r, lane);
  const int k = l.k;
  const bool mine = l.active && l.part == 0;
  const int w_begin = static_cast<int>(static_cast<long long>(blockIdx.x) * a_.W / gridDim.x);
  const int w_end = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * a_.W / gridDim.x);
  const int cols = min(l.rows, 8), chunks = l.rows / cols;               // columns of a table a lane sums at a time
  for (int w0 = w_begin; w0 < w_end; w0 += warps) {
    const int w = w0 + wib;
    if (w < w_end) {
      const float* g = a_.G + static_cast<size_t>(w) * n * r;
      const float* cw = a_.coeff + static_cast<size_t>(w) * n;
      const int* tg = a_.targets + static_cast<size_t>(w) * n;
      float* post = a_.post + static_cast<size_t>(w) * n * r;
      const float l0 = l.active ? a_.logw[static_cast<size_t>(w) * a_.sum_rows + k] : 0.f;
      // ---- forward
      float alpha = l.active ? l0 + g[k] : -CUDART_INF_F;
      float gi = l.active && n > 1 ? g[r + k] : 0.f;
      if (mine) us[k] = alpha;
      for (int i = 1; i < n; ++i) {
        const float g_next = l.active && i + 1 < n ? g[(i + 1) * r + k] : 0.f;
        float m;
        const float c = hmm_forward_sum<false>(alpha, ev + (i & 1) * 32, E + (i - 1) * rr, l, r, m);
        alpha = l.active ? m + __logf(c) + gi : -CUDART_INF_F;
        gi = g_next;
        if (mine) {
          us[i * (r + 1) + k] = alpha;
          xs[i * r + k] = c;
        }
      }
      __syncwarp();
      // ---- every prefix, lane = slot; its log-sum-exp is kept by the lane (slots past 32: read back)
      float lp_mine = 0.f;
      for (int i = lane; i < n; i += 32) {
        const float lp = thread_lse(us + i * (r + 1), r);
        a_.prefix[static_cast<size_t>(w) * n + i] = lp;
        if (i < 32) lp_mine = lp;
      }
      __syncwarp();
      auto prefix_of = [&](int i) { return i < 32 ? __shfl_sync(kFull, lp_mine, i) : a_.prefix[static_cast<size_t>(w) * n + i]; };
      // ---- reverse sweep
      const float lp_last = prefix_of(n - 1);
      float al_i = alpha;                                                // alpha_i of the lane's state
      float abar = l.active ? cw[n - 1] * __expf(alpha - lp_last) : 0.f;
      for (int i = n - 1; i >= 1; --i) {
        const float al = l.active ? us[(i - 1) * (r + 1) + k] : -CUDART_INF_F;
        const float lp = prefix_of(i - 1);
        float m = warp_max_nan(al);
        if (m == -CUDART_INF_F) m = 0.f;
        const float u = __expf(al - m);
        const float c = mine ? xs[i * r + k] : 1.f;                      // (one lane of a state reads its sum and puts x in its place)
        const bool tiny = sum_lost(c, abar);
        if (mine) {
          post[static_cast<size_t>(i) * r + k] = tg[i] >= 0 ? abar : 0.f;
          xs[i * r + k] = tiny ? 0.f : __fdividef(abar, c);
        }
        unsigned lost = __ballot_sync(kFull, tiny && abar != 0.f);
        __syncwarp();
        float prop = 0.f;
        const float* row = E + (i - 1) * rr + k * r;
        const float* x = xs + i * r;
        if (l.rows == 32) {                                              // float4 reads rotated by the lane: conflict-free
          const float4 *row4 = reinterpret_cast<const float4*>(row), *x4 = reinterpret_cast<const float4*>(x);
          float p1 = 0.f, p2 = 0.f, p3 = 0.f;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int j = (q + lane) & 7;
            const float4 a = row4[j], y = x4[j];
            prop = fmaf(a.x, y.x, prop);
            p1 = fmaf(a.y, y.y, p1);
            p2 = fmaf(a.z, y.z, p2);
            p3 = fmaf(a.w, y.w, p3);
          }
          prop = (prop + p1) + (p2 + p3);
        } else if (l.active) {
          for (int q = 0; q < l.rows; ++q) {
            const int b = l.part * l.rows + ((q + k) & (l.rows - 1));
            prop = fmaf(row[b], x[b], prop);
          }
        }
        for (int off = r; off < r * l.parts; off <<= 1) prop += __shfl_xor_sync(kFull, prop, off);
        prop *= u;
        if (lost != 0) {                                                 // columns left out above
          const float back = l.active && al_i != -CUDART_INF_F ? g[i * r + k] - al_i : -CUDART_INF_F;
          prop += hmm_lost_columns(lost, al, back, abar, logA + (i - 1) * rr + k * r, dT + (i - 1) * rr + k * r, mine);
        }
        if (mine) {
          us[(i - 1) * (r + 1) + k] = u;
          props[i * r + k] = prop;
        }
        abar = l.active ? cw[i - 1] * __expf(al - lp) + prop : 0.f;
        al_i = al;
      }
      float total = mine ? abar : 0.f;                                   // sum_z abar_0[z]
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) total += __shfl_xor_sync(kFull, total, off);
      if (mine) {
        post[k] = tg[0] >= 0 ? abar : 0.f;
        a_.dsum[static_cast<size_t>(w) * a_.dsum_pitch + k] = __float2bfloat16_rn(abar - __expf(l0) * total);
      }
    }
    __syncthreads();
    // ---- the batch's rank-one terms
    const int count = min(warps, w_end - w0);
    for (int task = wib; task < (n - 1) * chunks; task += warps) {
      const int i = 1 + task / chunks, b0 = l.part * l.rows + (task % chunks) * cols;
      if (!l.active) continue;
      float* sum = acc + (i - 1) * rr + b0 * r + k;
      float s[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) s[q] = q < cols ? sum[q * r] : 0.f;
      const float* from = area;
      if (cols == 8) {
#pragma unroll 2
        for (int j = 0; j < count; ++j, from += warp_floats) {
          const float u = from[off_u + (i - 1) * (r + 1) + k], pr = -from[off_prop + i * r + k];
          const float4 x0 = *reinterpret_cast<const float4*>(from + i * r + b0), x1 = *reinterpret_cast<const float4*>(from + i * r + b0 + 4);
          s[0] += fmaf(u, x0.x, pr);
          s[1] += fmaf(u, x0.y, pr);
          s[2] += fmaf(u, x0.z, pr);
          s[3] += fmaf(u, x0.w, pr);
          s[4] += fmaf(u, x1.x, pr);
          s[5] += fmaf(u, x1.y, pr);
          s[6] += fmaf(u, x1.z, pr);
          s[7] += fmaf(u, x1.w, pr);
        }
      } else {
        for (int j = 0; j < count; ++j, from += warp_floats) {
          const float u = from[off_u + (i - 1) * (r + 1) + k], pr = -from[off_prop + i * r + k];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < cols) s[q] += fmaf(u, from[i * r + b0 + q], pr);
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < cols) sum[q * r] = s[q];
    }
    __syncthreads();                                                     // the warps' vectors are reused by the next batch
  }
  // ---- dT += A * (the running sums), four adjacent entries at a time where dT is aligned for it
  if (rr % 4 == 0 && (reinterpret_cast<uintptr_t>(dT) & 15u) == 0) {
    for (int e = threadIdx.x * 4; e < tables; e += blockDim.x * 4) {
      const int q = e % rr, a = q / r, b = q - a * r;                    // (r a power of two: four entries of one row, or whole rows)
      float v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int at = (a * r + b + t) / r, bt = (b + t) % r;
        v[t] = E[e + t] * acc[(e - q) + bt * r + at];
      }
      if (!(v[0] == 0.f && v[1] == 0.f && v[2] == 0.f && v[3] == 0.f))
        atomicAdd(reinterpret_cast<float4*>(dT + e), make_float4(v[0], v[1], v[2], v[3]));
    }
  } else {
    for (int e = threadIdx.x; e < tables; e += blockDim.x) {
      const int q = e % rr, a = q / r, b = q - a * r;
      const float v = E[e] * acc[(e - q) + b * r + a];
      if (v != 0.f) atomicAdd(dT + e, v);
    }
  }
}

// ---------------------------------------------------------------- circuit backward: binary tree (Eq. BTree)
// Upward pass as in circuit_btree_kernel (prod[j][z], S[c][z]); downward pass with U[j][z] = log-weight of everything
// outside node j's subtree given z_j = z: U[0] = log omega_root, U[c][b] = LSE_z(U[j][z] + S[sibling][z] + logOmega_c[z][b]).
// Posterior of a latent: gamma_j = exp(U[j] + prod[j] - log q); a token's evidence gradient is its owner's gamma.
// Pairwise posterior xi_c[z][b] = exp(U[j][z] + S[sib][z] + logOmega_c[z][b] + prod[c][b] - log q); through the row
// softmax: xi_c[z][b] - Omega_c[z][b] gamma_j[z]. The tables are streamed twice (up: deepest parents first; down: in
// address order). Shared memory per warp: 3*(n-1)*r + 2*r*r + 32 floats.  r <= 32.
__host__ __device__ inline size_t btree_backward_warp_floats(int n, int r) {
  return 3 * static_cast<size_t>(n - 1) * r + 2 * static_cast<size_t>(r) * r + 32;
}

__global__ void circuit_btree_backward_kernel(const CircuitBackwardArgs a_, unsigned* work_counter) {
  grid_launch_dependents();
  grid_dependency_wait();
  extern __shared__ __align__(16) float sm[];
  const int wib = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int n = a_.n, r = a_.r;
  float* prod = sm + static_cast<size_t>(wib) * btree_backward_warp_floats(n, r);
  float* S = prod + (n - 1) * r;
  float* U = S + (n - 1) * r;
  float* tabs = U + (n - 1) * r;
  float* cur = tabs + 2 * r * r;
  const bool has = lane < r;
  const int first_leaf_node = n / 2 - 1;
  const int rr = r * r;
  const int ntab = n - 2;
  auto child_of = [&](int t) { return 2 * (first_leaf_node - 1 - (t >> 1)) + 1 + (t & 1); };
  for (int w = next_window(work_counter, lane); w < a_.W; w = next_window(work_counter, lane)) {
    const float* g = a_.G + static_cast<size_t>(w) * n * r;
    const float* lw = a_.logw + static_cast<size_t>(w) * a_.sum_rows;
    const size_t drow = static_cast<size_t>(w) * a_.dsum_pitch;
    const float wt = a_.weight[w];
    // ---- upward
    for (int j = n - 2; j >= first_leaf_node; --j) {
      const int t0 = 2 * (j - first_leaf_node);
      if (has) prod[j * r + lane] = g[t0 * r + lane] + g[(t0 + 1) * r + lane];
    }
    if (ntab > 0) warp_table_load_async(tabs, lw + r + static_cast<size_t>(child_of(0) - 1) * rr, rr, lane);
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
      __syncwarp();
      const float sc = sum_layer_staged(tabs + (t & 1) * rr, prod + c * r, lane, r);
      if (has) S[c * r + lane] = sc;
      acc += sc;
      if (t & 1) {
        if (has) prod[((c - 2) >> 1) * r + lane] = acc;
        acc = 0.f;
      }
      __syncwarp();
    }
    const float logq = warp_lse(has ? lw[lane] + prod[lane] : 0.f, has);
    if (lane == 0 && a_.out != nullptr) a_.out[w] = logq;
    // ---- downward, children c = 1 .. n-2 in address order
    if (has) {
      U[lane] = lw[lane];
      a_.dsum[drow + lane] = __float2bfloat16_rn(wt * (__expf(lw[lane] + prod[lane] - logq) - __expf(lw[lane])));
    }
    if (ntab > 0) warp_table_load_async(tabs, lw + r, rr, lane);
    __syncwarp();
    for (int c = 1; c <= ntab; ++c) {
      const int j = (c - 1) >> 1;
      const int sib = (c & 1) ? c + 1 : c - 1;
      if (c < ntab) {
        warp_table_load_async(tabs + (c & 1) * rr, lw + r + static_cast<size_t>(c) * rr, rr, lane);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      if (has) cur[lane] = U[j * r + lane] + S[sib * r + lane];          // in[z]
      __syncwarp();
      const float* tab = tabs + ((c - 1) & 1) * rr;
      if (has) {
        // message to the child: lane b, over the parent's values z (column of the table)
        float m = -CUDART_INF_F;
        for (int z = 0; z < r; ++z) m = fmaxf(m, cur[z] + tab[z * r + lane]);
        float s = 0.f;
        for (int z = 0; z < r; ++z) s += __expf(cur[z] + tab[z * r + lane] - m);
        U[c * r + lane] = (m == -CUDART_INF_F) ? -CUDART_INF_F : m + __logf(s);
        // gradient of the child's table: lane z (row), over the child's values b
        const float in_z = cur[lane];
        const float gam_parent = __expf(U[j * r + lane] + prod[j * r + lane] - logq);
        const size_t off = static_cast<size_t>(r) + static_cast<size_t>(c - 1) * rr + lane * r;
        row_grad(tab + lane * r, prod + c * r, in_z - logq, gam_parent, wt, lane, r, a_.dsum + drow + off, nullptr);
      }
      __syncwarp();
    }
    // ---- evidence gradients: token i under its owner's posterior
    for (int i = 0; i < n; ++i) {
      const int o = first_leaf_node + (i >> 1);
      const bool valid = a_.targets[static_cast<size_t>(w) * n + i] >= 0;
      if (has)
        a_.post[(static_cast<size_t>(w) * n + i) * r + lane] = valid ? wt * __expf(U[o * r + lane] + prod[o * r + lane] - logq) : 0.f;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------- Eq. 6 through the binary tree in one sweep
// L = sum_j coeff_j log p_j. TreeSweep's upward and downward sweeps give every prefix log p_j from the messages S and D; the
// gradient is their reverse mode, in plain numbers of either sign (bounded by sum_j |coeff_j|):
//   owner of the tokens 2m, 2m+1, with rho_0 = softmax(D + G[2m]), rho_1 = softmax(D + G[2m] + G[2m+1]):
//     dD = c_{2m} rho_0 + c_{2m+1} rho_1, which also goes to G[2m]; c_{2m+1} rho_1 to G[2m+1];
//   back up the tree (reverse of the downward sweep): D_c[b] = LSE_z(in_c[z] + T_c[z][b]) gives
//     pd_c[z] = sum_b dD_c[b] exp(in_c[z] + T_c[z][b] - D_c[b]), dD of the parent = the sum over its two children, and pd of a
//     right child is also the gradient of its left sibling's S;
//   down again (reverse of the upward sweep): dS_c = pd of the right sibling (left children) + dprod of the parent, and
//     S_c[z] = LSE_b(T_c[z][b] + prod_c[b]) gives dprod_c[b] = sum_z dS_c[z] exp(T_c[z][b] + prod_c[b] - S_c[z]), which reaches
//     the two tokens of an owner. Here both parts of dL/dT_c[z][b] are at hand; through the row softmax of the table's logits:
//     (its two summands) - exp(T_c[z][b]) (pd_c[z] + dS_c[z]).
// Four passes over a window's n - 2 tables, in shared memory as probabilities (TreeSweep), each table read from and its gradient written
// to HBM once, as bf16: with u = exp(in - max), e = exp(prod - max) and the sums of the two sweeps, every summand above is a product
// of numbers per row and per column with the table's entry, so no entry takes another exponential (six, with log tables). The n backward
// passes of the prefix lengths it replaces read and accumulated the window's 57 KB
// n times (2186 us at 4096 windows, n = 16, r = 32, plus 48 us zeroing and 184 us converting the fp32 accumulators and 313 us
// for the prefixes; this kernel on log tables, two CTAs an SM, did all of it in 498 us inside a training step; on probabilities, three
// CTAs an SM, in 211; HBM would take 80). One CTA per window, a warp per node of a level, as circuit_btree_prefix_kernel.
__host__ __device__ inline size_t btree_loss_smem_floats(int n, int r, int warps, bool tables_in_smem) {
  const size_t vr = (static_cast<size_t>(r) + 3) / 4 * 4;
  return btree_prefix_smem_floats(n, r, warps, tables_in_smem) +
         (3 * static_cast<size_t>(n - 1) + n / 2 + 4 * static_cast<size_t>(warps)) * vr;
}
template <int R>
__global__ void __launch_bounds__(256, 3) circuit_btree_loss_backward_kernel(const CircuitBackwardArgs a_, int tables_in_smem) {
  grid_launch_dependents();
  grid_dependency_wait();
  extern __shared__ __align__(16) float sm[];
  const int n = a_.n, r = R > 0 ? R : a_.r;
  TreeSweep<R> t;
  t.init(sm, n, r, tables_in_smem != 0);
  const int lane = t.lane, wib = t.wib, warps = t.warps, vr = t.vr;
  const bool has = lane < r;
  float* dD = t.after();                           // [n - 1][vr] gradient of D
  float* pd = dD + (n - 1) * vr;                   // [n - 1][vr] gradient of in_c, per parent value
  float* dP = pd + (n - 1) * vr;                   // [n - 1][vr] gradient of prod_c
  float* late = dP + (n - 1) * vr;                 // [n / 2][vr] c_{2m+1} rho_1
  float* vec = late + t.owners * vr + wib * 4 * vr;   // four vectors of this warp
  const int w0 = static_cast<int>(static_cast<long long>(blockIdx.x) * a_.W / gridDim.x);
  const int w1 = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * a_.W / gridDim.x);
  for (int w = w0; w < w1; ++w) {
    const float* cw = a_.coeff + static_cast<size_t>(w) * n;
    const int* tg = a_.targets + static_cast<size_t>(w) * n;
    __nv_bfloat16* drow = a_.dsum + static_cast<size_t>(w) * a_.dsum_pitch;
    t.load(a_.G + static_cast<size_t>(w) * n * r, a_.logw + static_cast<size_t>(w) * a_.sum_rows, true);
    t.up();
    t.down();
    for (int m = wib; m < t.owners; m += warps) {  // prefixes and the gradient of the owners' D
      const int o = t.first_leaf_node + m;
      const float d1 = has ? t.D[o * vr + lane] + t.gs[2 * m * vr + lane] : -CUDART_INF_F;
      const float d2 = has ? d1 + t.gs[(2 * m + 1) * vr + lane] : -CUDART_INF_F;
      const float p0 = warp_lse_nan(d1), p1 = warp_lse_nan(d2);
      if (lane == 0) {
        a_.prefix[static_cast<size_t>(w) * n + 2 * m] = p0;
        a_.prefix[static_cast<size_t>(w) * n + 2 * m + 1] = p1;
        if (a_.out != nullptr && m == t.owners - 1) a_.out[w] = p1;
      }
      if (has) {
        const float l = cw[2 * m + 1] * __expf(d2 - p1);
        late[m * vr + lane] = l;
        dD[o * vr + lane] = fmaf(cw[2 * m], __expf(d1 - p0), l);
      }
    }
    __syncthreads();
    for (int L = t.depth; L >= 1; --L) {           // reverse of the downward sweep
      for (int c = (1 << L) - 1 + wib; c <= (2 << L) - 2; c += warps) {
        float dd = 0.f, Dc = 0.f;
        if (has) {
          if (L < t.depth) dD[c * vr + lane] = pd[(2 * c + 1) * vr + lane] + pd[(2 * c + 2) * vr + lane];
          dd = dD[c * vr + lane];
          Dc = t.D[c * vr + lane];
        }
        const float in_z = has ? t.in_of(c) : 0.f;
        float m;
        const float u = t.scaled(in_z, m);
        const float sum = has ? __expf(Dc - m) : 1.f;                    // sum_z u[z] T_c[z][lane]
        const bool tiny = has && sum_lost(sum, dd);
        float* x = vec;                            // dD_c over that sum
        if (has) x[lane] = tiny ? 0.f : __fdividef(dd, sum);
        unsigned lost = __ballot_sync(kFull, tiny && dd != 0.f);
        __syncwarp();
        float acc = u * row_dot(t.table_of(c), x, lane, r);
        for (; lost != 0; lost &= lost - 1) {      // with logarithms
          const int b = __ffs(lost) - 1;
          const float dd_b = __shfl_sync(kFull, dd, b), D_b = __shfl_sync(kFull, Dc, b);
          if (has) acc = fmaf(dd_b, __expf(in_z + t.log_table(c)[lane * r + b] - D_b), acc);
        }
        if (has) pd[c * vr + lane] = acc;
        __syncwarp();
      }
      __syncthreads();
    }
    if (wib == 0) {                                // the root's logits
      if (t.depth > 0 && has) dD[lane] = pd[vr + lane] + pd[2 * vr + lane];
      float d0 = has ? dD[lane] : 0.f;
      float total = d0;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) total += __shfl_xor_sync(kFull, total, off);
      if (has) drow[lane] = __float2bfloat16_rn(d0 - __expf(t.lw[lane]) * total);
    }
    for (int L = 1; L <= t.depth; ++L) {           // reverse of the upward sweep, and the tables' gradients
      for (int c = (1 << L) - 1 + wib; c <= (2 << L) - 2; c += warps) {
        const bool edge = c == (2 << L) - 2;       // on the right edge: no S
        const int j = (c - 1) >> 1;
        const bool edge_parent = j == (1 << L) - 2;   // (the root included)
        float in_z = 0.f, Sz = 0.f, ds = 0.f, sumz = 0.f, prod = 0.f, Dc = 0.f, dDc = 0.f;
        if (has) {
          ds = edge ? 0.f : ((c & 1) ? pd[(c + 1) * vr + lane] : 0.f) + (edge_parent ? 0.f : dP[j * vr + lane]);
          in_z = t.in_of(c);
          sumz = pd[c * vr + lane] + ds;
          if (!edge) {
            Sz = t.S[c * vr + lane];
            prod = t.prod_of(c);
          }
          Dc = t.D[c * vr + lane];
          dDc = dD[c * vr + lane];
        }
        float mi, mp;
        const float u = t.scaled(in_z, mi);
        const float e = edge ? 0.f : t.scaled(prod, mp);
        const float below = has ? __expf(Dc - mi) : 1.f;                 // sum_z u[z] T_c[z][lane]
        const float across = has && !edge ? __expf(Sz - mp) : 1.f;       // sum_b T_c[lane][b] e[b]
        const bool tiny_b = has && sum_lost(below, dDc), tiny_z = has && !edge && sum_lost(across, ds);
        unsigned lost_b = __ballot_sync(kFull, tiny_b && dDc != 0.f), lost_z = __ballot_sync(kFull, tiny_z && ds != 0.f);
        __nv_bfloat16* dst = drow + r + static_cast<size_t>(c - 1) * r * r;
        // dL/dT_c[z][b] = T_c[z][b] (u[z] x[b] + y[z] e[b] - (pd + dS)[z]), x = dD / below, y = dS / across; dprod[b] = e[b] sum_z T y
        const float x = tiny_b ? 0.f : __fdividef(dDc, below), y = tiny_z ? 0.f : __fdividef(ds, across);
        float4* zv = reinterpret_cast<float4*>(vec);
        if (has) zv[lane] = make_float4(u, y, sumz, 0.f);
        __syncwarp();
        const float* tab = t.table_of(c);
        if (r == 32) {                           // a lane takes two columns of every other row: 4-byte stores
          const int half = lane >> 4, b = 2 * (lane & 15);
          const float x0 = __shfl_sync(kFull, x, b), x1 = __shfl_sync(kFull, x, b + 1);
          const float e0 = __shfl_sync(kFull, e, b), e1 = __shfl_sync(kFull, e, b + 1);
          float a0 = 0.f, a1 = 0.f;
#pragma unroll 8
          for (int q = 0; q < 16; ++q) {
            const int z = 2 * q + half;
            const float2 p = *reinterpret_cast<const float2*>(tab + z * 32 + b);
            const float4 f = zv[z];
            a0 = fmaf(p.x, f.y, a0);
            a1 = fmaf(p.y, f.y, a1);
            const float g0 = p.x * fmaf(f.y, e0, fmaf(f.x, x0, -f.z)), g1 = p.y * fmaf(f.y, e1, fmaf(f.x, x1, -f.z));
            *reinterpret_cast<__nv_bfloat162*>(dst + z * 32 + b) = __floats2bfloat162_rn(g0, g1);
          }
          a0 += __shfl_xor_sync(kFull, a0, 16);
          a1 += __shfl_xor_sync(kFull, a1, 16);
          if (half == 0) *reinterpret_cast<float2*>(dP + c * vr + b) = make_float2(a0 * e0, a1 * e1);
        } else if (has) {
          float a0 = 0.f;
          for (int z = 0; z < r; ++z) {
            const float p = tab[z * r + lane];
            const float4 f = zv[z];
            a0 = fmaf(p, f.y, a0);
            dst[z * r + lane] = __float2bfloat16_rn(p * fmaf(f.y, e, fmaf(f.x, x, -f.z)));
          }
          dP[c * vr + lane] = a0 * e;
        }
        if ((lost_b | lost_z) != 0) {              // columns and rows left out above: with logarithms, over what was stored
          const float* logt = t.log_table(c);
          __syncwarp();
          for (; lost_b != 0; lost_b &= lost_b - 1) {                    // lane = z
            const int b = __ffs(lost_b) - 1;
            const float D_b = __shfl_sync(kFull, Dc, b), dD_b = __shfl_sync(kFull, dDc, b), e_b = __shfl_sync(kFull, e, b);
            if (has)
              dst[lane * r + b] = __float2bfloat16_rn(fmaf(dD_b, __expf(in_z + logt[lane * r + b] - D_b), tab[lane * r + b] * fmaf(y, e_b, -sumz)));
          }
          __syncwarp();
          float more = 0.f;
          for (; lost_z != 0; lost_z &= lost_z - 1) {                    // lane = b
            const int z = __ffs(lost_z) - 1;
            const float S_z = __shfl_sync(kFull, Sz, z), ds_z = __shfl_sync(kFull, ds, z), in = __shfl_sync(kFull, in_z, z);
            if (has) {
              const float l = logt[z * r + lane], own = ds_z * __expf(l + prod - S_z);
              const float4 f = zv[z];
              const float up = tiny_b && dDc != 0.f ? dDc * __expf(in + l - Dc) : 0.f;
              dst[z * r + lane] = __float2bfloat16_rn(fmaf(tab[z * r + lane], fmaf(f.x, x, -f.z), own + up));
              more += own;
            }
          }
          if (has) dP[c * vr + lane] += more;
        }
        __syncwarp();
      }
      __syncthreads();
    }
    for (int m = wib; m < t.owners; m += warps) {  // evidence of the tokens 2m and 2m + 1
      const int o = t.first_leaf_node + m;
      if (has) {
        const float back = t.depth > 0 && m < t.owners - 1 ? dP[o * vr + lane] : 0.f;   // (the last owner is on the right edge)
        float* dst = a_.post + (static_cast<size_t>(w) * n + 2 * m) * r + lane;
        dst[0] = tg[2 * m] >= 0 ? dD[o * vr + lane] + back : 0.f;
        dst[r] = tg[2 * m + 1] >= 0 ? late[m * vr + lane] + back : 0.f;
      }
    }
    __syncthreads();                               // shared memory is reused by the next window
  }
}

// ---------------------------------------------------------------- gradient with respect to the emission logits
// dlogit[t, c] = post[t, u] * (onehot(target[t, i] == c - u v) - exp(logit[t, c] - lse[t, u])),  u = c / v = i r + k,
// from the logits and log-sum-exps the forward pass kept (padding columns hold -inf: no mass, zero gradient; a
// marginalised byte has no gradient). Written once, as bf16 rows [T, pitch]: both weight-sized GEMMs read this one
// matrix, d hidden along its rows (K-major) and dW down its columns (MN-major). One streaming pass: a thread converts
// 8 adjacent logits (two 16-byte loads, one 16-byte store); v is a multiple of 16, so they belong to one unit.
struct LogitGradArgs {
  const float* logits;       // [T, Nc], pitch Nc
  const float* lse;          // [T, n r]
  const float* post;         // [T, n r]
  const int* targets;        // [T, n]
  __nv_bfloat16* dlogit;     // [T, pitch]
  size_t pitch;
  int T, Nc, n, r, v;
};

__global__ void __launch_bounds__(256) logit_gradient_kernel(const LogitGradArgs a) {
  grid_dependency_wait();
  const int c = (blockIdx.x * 256 + threadIdx.x) * 8;
  if (c >= a.Nc) return;
  const int units = a.n * a.r;
  const int u = c / a.v;
  const int i = u / a.r;
  const int col_in_unit = c - u * a.v;
  for (int t = blockIdx.y; t < a.T; t += gridDim.y) {
    const int tgt = a.targets[static_cast<size_t>(t) * a.n + i];
    const size_t tu = static_cast<size_t>(t) * units + u;
    const float pst = tgt >= 0 ? a.post[tu] : 0.f;
    const float lse2 = a.lse[tu] * kLog2e;
    const float4* src = reinterpret_cast<const float4*>(a.logits + static_cast<size_t>(t) * a.Nc + c);
    const float4 x0 = __ldcs(src), x1 = __ldcs(src + 1);
    const float xs[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
    const int rel = tgt - col_in_unit;
    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      o[q] = __float2bfloat16_rn(pst * ((rel == q ? 1.f : 0.f) - fast_ex2(fmaf(xs[q], kLog2e, -lse2))));
    *reinterpret_cast<uint4*>(a.dlogit + static_cast<size_t>(t) * a.pitch + c) = *reinterpret_cast<const uint4*>(o);
  }
  grid_launch_dependents();
}

// ---------------------------------------------------------------- plain bf16 GEMM on the tcgen05 tensor cores
// C[M, N] (fp32, row-major, pitch ldc) = A[M, K] B[N, K]^T with bf16 operands read where they lie, in either
// orientation: K-major (K contiguous in memory: 64-element K boxes of up to 256 rows) or MN-major (the M / N index
// contiguous: 64 x 64 boxes, two for the 128 rows of A, up to four for the columns of B). Out-of-range rows and
// columns read as zero. The K axis may consist of up to three segments with a B matrix each (d hidden sums over the
// emission rows, or W_base and the adaptors B, and the sum-unit rows, which are separate matrices); A then continues at a_k0[i]. Same pipeline as the
// projection kernel: one persistent CTA per SM, warp 0 TMA producer, warp 1 MMA issuer (two TMEM slots), warps 2..5 epilogue
// (one thread per row, 16 fp32 columns per step). CTAS = 1: a CTA works alone (M = 128, N = TN). CTAS = 2: a cluster of two
// shares every MMA (cta_group::2, M = 256), each CTA staging its own 128 rows of A and half of the columns of B, so a third
// less data moves from L2 to shared memory per multiply-add; barriers as in the projection kernel.
// Split of the last round: tiles are dealt to the workers (CTAs or pairs) round by round, and the `tail_tiles` that do not
// fill a round are cut along K into `split` parts each, dealt part by part (workers that run together then walk the same K
// range of different tiles and share its operands through L2). The parts are written as fp32 tiles and split_reduce_kernel adds
// them up in K order, spread over the whole device. (Added up by the warp that arrives last, a few warps read every part alone:
// 12 tiles in 8 parts took 29 us where the uncut launch takes 19.) It matters where a contraction has few tiles: d hidden of
// 2005 positions is 96 pair tiles for 74 pairs (415 -> 271 us), of 4096 positions 192 (2945 -> 2480 us, pairs and cut together).
struct PlainGemmParams {
  CUtensorMap tm_a;      // K-major: A [M, K], box 64 (k) x 128; MN-major: A^T [K, M], box 64 (m) x 64 (k)
  CUtensorMap tm_b[3];   // per K segment. K-major: B [N, K], box 64 (k) x TN / CTAS; MN-major: B^T [K, N], box 64 (n) x 64 (k)
  int a_k0[3];           // K coordinate of A at which each segment starts (multiples of 8)
  int seg_kblocks[3];    // 64-wide K blocks per segment (0: unused; only trailing ones are)
  int M, N;
  int m_tiles, n_tiles;  // m_tiles: tiles of CTAS * 128 rows
  int stages, stage_bytes;
  int wide_stores;       // C and ldc allow 32-byte stores
  float* C;
  size_t ldc;
  // The rows from m_end[0] on go to C2, those from m_end[1] on to C3 (same pitch): the weight gradients of several matrices
  // whose logit gradients lie side by side are one launch, instead of small launches that each end in a partial round.
  float *C2, *C3;
  int m_end[2];
  // Instead of C (C == NULL): the result split into two bf16 halves, x = hi + lo, written as [M, N / split_k, 2, split_k]
  // (group g of split_k columns: hi at column (2 g) split_k, lo at (2 g + 1) split_k; split_k a multiple of 16).
  __nv_bfloat16* C_hilo;
  int split_k;
  // Instead of C (C == NULL, C_hilo == NULL): the result rounded to bf16, [M, N] at a pitch of ldc elements.
  __nv_bfloat16* C_bf16;
  // Several independent products of the same shape in one launch (batches > 1; one K segment): product q reads A at
  // its M / K coordinates plus q * a_m_step / q * a_k_step, B at its N / K coordinates plus q * b_n_step / q * b_k_step,
  // and writes at C (or C_bf16) + q * c_step elements. Rows of A and columns of B past M and N are then another product's
  // data, not zeros: they reach accumulator rows and columns that are not written. Along K the operands must agree on
  // zeros past the product's own extent (the caller pads one of them).
  int batches, a_m_step, a_k_step, b_n_step, b_k_step;
  size_t c_step;
  int tail_tiles, split;      // the last tail_tiles tiles are cut into `split` parts (1: not cut)
  float* partial;             // [tail_tiles][split][CTAS][4 warps] runs of 32 x TN floats, lane-fastest
  unsigned* status;
  uint64_t wait_limit_ns;   // limit of every pipeline wait
};
constexpr int kPlainTileN = 256;
constexpr uint32_t kMnBoxBytes = 64 * kBlockK * 2;   // one 64 x 64 bf16 box: 8 KB
// Scratch of a split launch: parts of at most kSplitParts 128 x 256 tiles (three rounds of a 148-SM device).
constexpr int kSplitParts = 444;
constexpr size_t kSplitPartBytes = static_cast<size_t>(kBlockM) * kPlainTileN * sizeof(float);

// Work item `item` of a launch: the tile and the K blocks [kb0, kb1) of it; tail >= 0: index of the cut tile, part its part.
struct PlainItem {
  int bt, mt, nt, kb0, kb1, tail, part;
};
__device__ __forceinline__ PlainItem plain_item(const PlainGemmParams& p, int item, int kblocks) {
  PlainItem w;
  const int per_batch = p.m_tiles * p.n_tiles;
  const int whole = per_batch * p.batches - p.tail_tiles;
  int tile = item;
  w.tail = -1;
  w.part = 0;
  w.kb0 = 0;
  w.kb1 = kblocks;
  if (item >= whole) {
    const int q = item - whole;
    w.part = q / p.tail_tiles;
    w.tail = q - w.part * p.tail_tiles;
    tile = whole + w.tail;
    w.kb0 = static_cast<int>(static_cast<long long>(w.part) * kblocks / p.split);
    w.kb1 = static_cast<int>(static_cast<long long>(w.part + 1) * kblocks / p.split);
  }
  // n-tile fastest: the CTAs running together cover a few m-tiles x all n-tiles, so the (larger) A operand is
  // streamed from HBM once and the B operand once per wave of m-tiles
  w.bt = tile / per_batch;
  const int rest = tile - w.bt * per_batch;
  w.nt = rest % p.n_tiles;
  w.mt = rest / p.n_tiles;
  return w;
}

// First element of a row of the fp32 result (row < M).
__device__ __forceinline__ float* plain_row(const PlainGemmParams& p, int row) {
  if (row < p.m_end[0]) return p.C + static_cast<size_t>(row) * p.ldc;
  if (row < p.m_end[1]) return p.C2 + static_cast<size_t>(row - p.m_end[0]) * p.ldc;
  return p.C3 + static_cast<size_t>(row - p.m_end[1]) * p.ldc;
}
// Sixteen adjacent columns of one row of the result, in whichever form it is wanted. crow: where the row starts in C;
// coff: its offset in C_bf16.
__device__ __forceinline__ void plain_store16(const PlainGemmParams& p, const float (&x)[16], int row, float* crow, size_t coff, int col0) {
  if (p.C == nullptr && p.C_hilo == nullptr) {
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) o[q] = __float2bfloat16_rn(x[q]);
    uint4* dst = reinterpret_cast<uint4*>(p.C_bf16 + coff + col0);      // ldc, c_step and C_bf16 keep 16 columns 32-byte aligned
    dst[0] = reinterpret_cast<const uint4*>(o)[0];
    dst[1] = reinterpret_cast<const uint4*>(o)[1];
  } else if (p.C == nullptr) {
    // 16 columns of one group: 32 bytes of high halves and 32 bytes of low halves
    const int grp = col0 / p.split_k, q0 = col0 - grp * p.split_k;
    __align__(16) __nv_bfloat16 hi[16], lo[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      hi[q] = __float2bfloat16_rn(x[q]);
      lo[q] = __float2bfloat16_rn(x[q] - __bfloat162float(hi[q]));
    }
    __nv_bfloat16* dst = p.C_hilo + static_cast<size_t>(row) * (2 * p.N) + static_cast<size_t>(2 * grp) * p.split_k + q0;
    reinterpret_cast<uint4*>(dst)[0] = reinterpret_cast<const uint4*>(hi)[0];
    reinterpret_cast<uint4*>(dst)[1] = reinterpret_cast<const uint4*>(hi)[1];
    reinterpret_cast<uint4*>(dst + p.split_k)[0] = reinterpret_cast<const uint4*>(lo)[0];
    reinterpret_cast<uint4*>(dst + p.split_k)[1] = reinterpret_cast<const uint4*>(lo)[1];
  } else if (p.wide_stores) {                    // 32-byte aligned rows: one full sector per store
    st_global_v8(crow + col0, x);
    st_global_v8(crow + col0 + 8, x + 8);
  } else {
    float4* c4 = reinterpret_cast<float4*>(crow + col0);
#pragma unroll
    for (int q = 0; q < 4; ++q) c4[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
  }
}

// TN: columns of an accumulator tile: 256, or 64 for the batched products whose N is a rank (MN-major B only: the boxes
// of the tensor map are 64 wide) - what is fetched, multiplied and read back for columns that do not exist is a quarter.
template <bool A_MN, bool B_MN, int TN = 256, int CTAS = 1>
__global__ void __launch_bounds__(kGemmThreads, 1) plain_gemm_kernel(const __grid_constant__ PlainGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* tiles = smem_raw + (tiles_addr - raw_addr);
  GemmControl* ctl = reinterpret_cast<GemmControl*>(tiles + static_cast<size_t>(p.stages) * p.stage_bytes);
  const int warp = static_cast<int>(warp_uniform(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const int kblocks = p.seg_kblocks[0] + p.seg_kblocks[1] + p.seg_kblocks[2];
  const int num_items = p.m_tiles * p.n_tiles * p.batches + p.tail_tiles * (p.split - 1);
  const uint32_t cta_rank = CTAS == 2 ? warp_uniform(cluster_cta_rank()) : 0u;      // 0 = the pair's leader
  const int first_item = CTAS == 2 ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int item_step = CTAS == 2 ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);
  constexpr uint32_t kSlots = 2;
  constexpr int kBCols = TN / CTAS;                                   // columns of B this CTA stages
  constexpr uint32_t kBBytes = kBCols * kBlockK * 2;
  static_assert(CTAS == 1 || TN == kPlainTileN, "pairs share 256-column tiles");

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (uint32_t s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&ctl->tfull[s]), 1);
      mbar_init(smem_u32(&ctl->tempty[s]), 4 * CTAS);
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    ctl->wait_limit_ns = p.wait_limit_ns;
    fence_mbar_init();
    tma_prefetch_desc(&p.tm_a);
    tma_prefetch_desc(&p.tm_b[0]);
    if (p.seg_kblocks[1] > 0) tma_prefetch_desc(&p.tm_b[1]);
    if (p.seg_kblocks[2] > 0) tma_prefetch_desc(&p.tm_b[2]);
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
  grid_launch_dependents();            // the next kernel's CTAs may be scheduled as SMs free up
  grid_dependency_wait();

  if (warp == 0) {
    // One K block must be asked for in less time than its MMAs take (256 cycles), so that little is computed per block.
    // Weight gradients of few positions in pairs are bound by their fp32 stores, and this warp waits most of the time: then one lane does. As a whole warp /
    // so / issued from lane 0's own branch, us: dW_emit of 8 x 16 x 320, d = 4096 from 60 positions 192 / 166 / 168, 250 208 / 186 / 195, 500 232 / 213 / 224, 1000
    // (16 K blocks) 293 / 281 / 294; but 1100 319 / 317 / 311, 1500 371 / 381 / 372, 4096 906 / 935 / 935. Lone CTAs, 8 x 8 x 256, d = 2048, 900 positions
    // 58 / 61 / 62; K-major operands (long K) 250 positions 75 / 78 / 79.
    const bool few_blocks = A_MN && CTAS == 2 && kblocks <= 16;
    const uint32_t lead = elect_one(), expects = cta_rank == 0 ? lead : 0u;
    uint32_t stage = 0, phase = 0, issued = 0;
    bool ok = true;
    auto load = [&](uint32_t dst, const CUtensorMap* tm, uint32_t full, int x, int y) {
      if (CTAS == 2) tma_load_2d_pair(lead, dst, tm, full, x, y);
      else tma_load_2d(lead, dst, tm, full, x, y);
    };
    const uint32_t own_full = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    const uint32_t full0 = CTAS == 2 ? warp_uniform(cluster_map_shared(own_full, 0)) : own_full;   // the leader's barriers
    for (int item = first_item; item < num_items && ok; item += item_step) {
      const PlainItem w = plain_item(p, item, kblocks);
      const int am = (w.mt * CTAS + static_cast<int>(cta_rank)) * kBlockM + w.bt * p.a_m_step;   // this CTA's rows of A,
      const int bn = w.nt * TN + static_cast<int>(cta_rank) * kBCols + w.bt * p.b_n_step;        // its columns of B
      int kb = w.kb0, seg_begin = 0;
      for (int seg = 0; seg < 3 && ok; ++seg) {
        const int seg_end = seg_begin + p.seg_kblocks[seg], stop = min(seg_end, w.kb1);
        const CUtensorMap* tm_b = &p.tm_b[seg];
        int ak = p.a_k0[seg] + (kb - seg_begin) * kBlockK + w.bt * p.a_k_step, bk = (kb - seg_begin) * kBlockK + w.bt * p.b_k_step;
        for (; kb < stop; ++kb, ak += kBlockK, bk += kBlockK) {
          ok = few_blocks ? bounded_wait_warp(empty0 + 8 * stage, phase ^ 1u, ctl, p.status, lane) : bounded_wait_all(empty0 + 8 * stage, phase ^ 1u, ctl, p);
          if (!ok) break;
          const uint32_t full = full0 + 8 * stage, a_dst = tiles_addr + stage * p.stage_bytes;
          mbar_arrive_expect_tx(expects, own_full + 8 * stage, CTAS * (kABytes + kBBytes));      // of both CTAs' copies when paired
          if (A_MN) {
#pragma unroll
            for (int q = 0; q < kBlockM / 64; ++q) load(a_dst + q * kMnBoxBytes, &p.tm_a, full, am + q * 64, ak);
          } else {
            load(a_dst, &p.tm_a, full, ak, am);
          }
          if (B_MN) {
#pragma unroll
            for (int q = 0; q < kBCols / 64; ++q) load(a_dst + kABytes + q * kMnBoxBytes, tm_b, full, bn + q * 64, bk);
          } else {
            load(a_dst + kABytes, tm_b, full, bk, bn);
          }
          ++issued;
          if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
        seg_begin = seg_end;
      }
    }
    // no copy may still be in flight when the CTA goes away (they have all landed unless some warp gave up)
    if (CTAS == 1 || cta_rank == 0) {
      for (uint32_t s = 0; s < static_cast<uint32_t>(p.stages) && s < issued; ++s)
        drain_wait(own_full + 8 * s, ((issued - 1 - s) / p.stages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (cta_rank == 0) {
      const uint32_t lead = elect_one();
      uint32_t stage = 0, phase = 0, use = 0;
      bool ok = first_item >= num_items || first_wait(smem_u32(&ctl->full[0]), ctl, p);
      const uint32_t idesc = umma_idesc_bf16(kBlockM * CTAS, TN, A_MN, B_MN);
      // descriptor advance per K=16 step, in 16-byte units: 32 bytes along a swizzled K-major row, two 8-row groups
      // (2048 bytes) down an MN-major box
      constexpr uint32_t kStepA = A_MN ? 128u : 2u, kStepB = B_MN ? 128u : 2u;
      const uint64_t a_desc0 = A_MN ? umma_smem_desc_mn_sw128(tiles_addr, kMnBoxBytes) : umma_smem_desc_sw128(tiles_addr);
      const uint64_t b_desc0 = B_MN ? umma_smem_desc_mn_sw128(tiles_addr + kABytes, kMnBoxBytes)
                                    : umma_smem_desc_sw128(tiles_addr + kABytes);
      const uint32_t stage_step = p.stage_bytes >> 4, full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
      auto commit = [&](uint32_t bar) {                        // pairs: in both CTAs
        if (CTAS == 2) umma_commit_pair(lead, bar);
        else umma_commit(lead, bar);
      };
      for (int item = first_item; item < num_items && ok; item += item_step, ++use) {
        const PlainItem w = plain_item(p, item, kblocks);
        const uint32_t slot = use % kSlots;
        if (!bounded_wait_all(smem_u32(&ctl->tempty[slot]), ((use / kSlots) & 1u) ^ 1u, ctl, p)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + slot * TN;
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          if (!bounded_wait_all(full0 + 8 * stage, phase, ctl, p)) { ok = false; break; }
          tc_fence_after();
          const uint64_t a_desc = a_desc0 + stage * stage_step, b_desc = b_desc0 + stage * stage_step;
#pragma unroll
          for (int kk = 0; kk < kBlockK / 16; ++kk) {
            const uint32_t acc = (kb != w.kb0 || kk != 0) ? 1u : 0u;
            if (CTAS == 2) umma_bf16_pair(lead, d_tmem, a_desc + kStepA * kk, b_desc + kStepB * kk, idesc, acc);
            else umma_bf16(lead, d_tmem, a_desc + kStepA * kk, b_desc + kStepB * kk, idesc, acc);
          }
          commit(empty0 + 8 * stage);
          if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        commit(smem_u32(&ctl->tfull[slot]));
      }
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    uint32_t use = 0;
    for (int item = first_item; item < num_items; item += item_step, ++use) {
      const PlainItem w = plain_item(p, item, kblocks);
      const uint32_t slot = use % kSlots;
      if (!bounded_wait_warp(smem_u32(&ctl->tfull[slot]), (use / kSlots) & 1u, ctl, p.status, lane)) break;
      tc_fence_after();
      const int row = (w.mt * CTAS + static_cast<int>(cta_rank)) * kBlockM + quarter * 32 + lane;
      const uint32_t tcol = lane_base + slot * TN;
      const size_t coff = static_cast<size_t>(row < p.M ? row : 0) * p.ldc + static_cast<size_t>(w.bt) * p.c_step;
      float* crow = p.C == nullptr || row >= p.M ? nullptr : plain_row(p, row) + static_cast<size_t>(w.bt) * p.c_step;
      const int batches = min(TN, p.N - w.nt * TN) / 16;         // (N is a multiple of 16) the rest lies past the last column
      const bool cut = w.tail >= 0;
      // a cut tile's part: 32 x TN floats per warp, lane-fastest so that every access is 512 contiguous bytes
      float4* part = reinterpret_cast<float4*>(p.partial) +
                     (cut ? (((static_cast<size_t>(w.tail) * p.split + w.part) * CTAS + cta_rank) * 4 + quarter) * (8 * TN) : 0) + lane;
      for (int b = 0; b < batches; ++b) {
        float x[16];
        tmem_ld16(tcol + b * 16, x);
        if (cut) {
#pragma unroll
          for (int q = 0; q < 4; ++q) part[b * 128 + 32 * q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
        } else if (row < p.M) {
          plain_store16(p, x, row, crow, coff, w.nt * TN + b * 16);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CTAS == 2) mbar_arrive_cluster(cluster_map_shared(smem_u32(&ctl->tempty[slot]), 0));
        else mbar_arrive(smem_u32(&ctl->tempty[slot]));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) drain_after_abort<CTAS>(ctl, cta_rank == 0);
  if (CTAS == 2) {        // a CTA of a pair may leave only when its partner no longer needs it
    __syncthreads();
    cluster_sync_all();
  }
  if (warp == 1) {
    tc_fence_after();
    if (CTAS == 2) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// The cut tiles of a plain GEMM (256-column tiles, one product): adds their parts up in K order and stores the result. One
// warp per 32 rows x 16 columns; grid.x = tail_tiles * ctas * 8, 8 warps.
__global__ void __launch_bounds__(256) split_reduce_kernel(const __grid_constant__ PlainGemmParams p, int ctas) {
  grid_dependency_wait();   // the parts come from the kernel before this one
  const int lane = threadIdx.x & 31;
  int q = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int b = q & 15;
  q >>= 4;
  const int quarter = q & 3;
  q >>= 2;
  const int rank = q % ctas, tail = q / ctas;
  const int tile = p.m_tiles * p.n_tiles - p.tail_tiles + tail;
  const int nt = tile % p.n_tiles, mt = tile / p.n_tiles;
  const int row = (mt * ctas + rank) * kBlockM + quarter * 32 + lane, col0 = nt * kPlainTileN + b * 16;
  if (col0 >= p.N) return;
  const size_t pitch = static_cast<size_t>(ctas) * 4 * (8 * kPlainTileN);
  const float4* src = reinterpret_cast<const float4*>(p.partial) + static_cast<size_t>(tail) * p.split * pitch +
                      (static_cast<size_t>(rank) * 4 + quarter) * (8 * kPlainTileN) + b * 128 + lane;
  float x[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) x[e] = 0.f;
#pragma unroll 4
  for (int part = 0; part < p.split; ++part) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 y = src[part * pitch + 32 * e];
      x[4 * e] += y.x;
      x[4 * e + 1] += y.y;
      x[4 * e + 2] += y.z;
      x[4 * e + 3] += y.w;
    }
  }
  if (row < p.M) plain_store16(p, x, row, p.C == nullptr ? nullptr : plain_row(p, row), static_cast<size_t>(row) * p.ldc, col0);
  grid_launch_dependents();
}

}  // namespace mtpc
