// Sorting of the rejected windows of a long draft by the slot of their first rejected byte (Algorithm 3), for drafts whose
// logits did not fit the workspace: the acceptance stage recomputes that slot's logits. A counting sort over the n slots packs
// the hidden states of the windows that share a slot into consecutive rows of a staging buffer, so that one pass of the
// projection kernel multiplies each by the r units of its slot only.
//   group_count_kernel   histogram of the windows over the slots
//   group_scan_kernel    exclusive scan -> first staging row of every slot, and the list of 128-row tiles
//   group_gather_kernel  every window takes the next free row of its slot and copies its hidden state there
// The order inside a slot depends on the order of the atomic increments; nothing downstream depends on it.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace mtpc {

constexpr int kGroupThreads = 256;
constexpr int kGroupScanThreads = 1024;

// One tile of the sorted pass: `count` <= 128 staging rows starting at `row0`, all of slot `unit`.
struct GroupTile {
  int unit, row0, count, pad;
};

// counts[slot] += 1 for every window rejected in that slot (first_rejected[w] = -1: none). Shared-memory histogram per CTA,
// flushed once.
__global__ void __launch_bounds__(kGroupThreads) group_count_kernel(const int* __restrict__ first_rejected,
                                                                    int* __restrict__ counts, int windows, int slots) {
  extern __shared__ int hist[];
  for (int k = threadIdx.x; k < slots; k += kGroupThreads) hist[k] = 0;
  __syncthreads();
  for (int w = blockIdx.x * kGroupThreads + threadIdx.x; w < windows; w += gridDim.x * kGroupThreads) {
    const int s = first_rejected[w];
    if (s >= 0) atomicAdd(&hist[s], 1);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < slots; k += kGroupThreads)
    if (hist[k]) atomicAdd(&counts[k], hist[k]);
}

// One CTA. offsets[u] = number of windows in the slots before u; tiles = every slot cut into runs of <= 128 rows, in slot
// order; *num_tiles = how many. Thread t owns the slots [t * per, (t + 1) * per).
__global__ void __launch_bounds__(kGroupScanThreads) group_scan_kernel(const int* __restrict__ counts,
                                                                       int* __restrict__ offsets,
                                                                       GroupTile* __restrict__ tiles,
                                                                       int* __restrict__ num_tiles, int units) {
  __shared__ int warp_rows[kGroupScanThreads / 32], warp_tiles[kGroupScanThreads / 32];
  const int per = (units + kGroupScanThreads - 1) / kGroupScanThreads;
  const int u0 = threadIdx.x * per;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int rows = 0, ntl = 0;
  for (int q = 0; q < per; ++q) {
    const int c = (u0 + q < units) ? counts[u0 + q] : 0;
    rows += c;
    ntl += (c + 127) >> 7;
  }
  // inclusive scan of (rows, tiles) over the CTA: within the warp by shuffles, across warps through shared memory
  int rs = rows, ts = ntl;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, rs, off);
    const int b = __shfl_up_sync(0xffffffffu, ts, off);
    if (lane >= off) { rs += a; ts += b; }
  }
  if (lane == 31) { warp_rows[warp] = rs; warp_tiles[warp] = ts; }
  __syncthreads();
  if (warp == 0) {
    int a = warp_rows[lane], b = warp_tiles[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, a, off);
      const int y = __shfl_up_sync(0xffffffffu, b, off);
      if (lane >= off) { a += x; b += y; }
    }
    warp_rows[lane] = a;
    warp_tiles[lane] = b;
    if (lane == 31) *num_tiles = b;
  }
  __syncthreads();
  int row = rs - rows + (warp ? warp_rows[warp - 1] : 0);     // exclusive prefix of this thread's first unit
  int tile = ts - ntl + (warp ? warp_tiles[warp - 1] : 0);
  for (int q = 0; q < per; ++q) {
    const int u = u0 + q;
    if (u >= units) break;
    const int c = counts[u];
    offsets[u] = row;
    for (int done = 0; done < c; done += 128) {
      GroupTile t;
      t.unit = u;
      t.row0 = row + done;
      t.count = c - done < 128 ? c - done : 128;
      t.pad = 0;
      tiles[tile++] = t;
    }
    row += c;
  }
}

// One warp per window: lane 0 takes the next free staging row of the slot the window was rejected in and records it (row_of), the
// warp copies the hidden state of the window's position (d bf16, d a multiple of 8, rows 16-byte aligned) there.
__global__ void __launch_bounds__(kGroupThreads) group_gather_kernel(const int* __restrict__ first_rejected,
                                                                     const __nv_bfloat16* __restrict__ hidden,
                                                                     const int* __restrict__ offsets,
                                                                     int* __restrict__ cursors,
                                                                     __nv_bfloat16* __restrict__ stage, int windows, int wpp,
                                                                     int d, int* __restrict__ row_of) {
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (kGroupThreads / 32);
  const int vecs = d / 8;                                      // 16-byte pieces per row
  for (int w = blockIdx.x * (kGroupThreads / 32) + (threadIdx.x >> 5); w < windows; w += warps) {
    const int s = first_rejected[w];
    if (s < 0) continue;                                       // warp-uniform: the whole warp reads the same entry
    int row = 0;
    if (lane == 0) {
      row = offsets[s] + atomicAdd(&cursors[s], 1);
      row_of[w] = row;
    }
    row = __shfl_sync(0xffffffffu, row, 0);
    const uint4* src = reinterpret_cast<const uint4*>(hidden + static_cast<size_t>(w / wpp) * d);
    uint4* dst = reinterpret_cast<uint4*>(stage + static_cast<size_t>(row) * d);
    for (int q = lane; q < vecs; q += 32) dst[q] = src[q];
  }
}

}  // namespace mtpc
