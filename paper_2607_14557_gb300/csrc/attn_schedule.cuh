// Work schedule of the 16-bit attention kernel: the code of one block, run by a
// kernel of its own or by an extra block of the layer's first norm.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace seer {

constexpr int kAttnRows = 128;     // query rows of a tile
constexpr int kAttnTiles = 2;      // query tiles of a unit

// One block: per-segment key counts -> work units (b, h, first q-tile, tiles)
// of up to NT query tiles, ordered by descending kv length so the longest
// segments start first.
// sh: 4 B ints of shared memory.
__device__ __forceinline__ void attn_schedule_block(const ScheduleArgs& a, int* err, int* sh) {
  const int *cu = a.cu, *cu_kv = a.cu_kv, *kv_len = a.kv_len;
  const int B = a.B, H = a.n_heads, T_cap = a.T_cap, max_units = a.max_units;
  int4* work = a.work;
  int* work_count = a.work_count;
  int* ntile = sh;           // [B]
  int* kvs = sh + B;         // [B]
  int* off = sh + 2 * B;     // [B]
  int* rank = sh + 3 * B;    // [B]
  for (int i = threadIdx.x; i < B; i += blockDim.x) {
    const int L = cu[i + 1] - cu[i];
    const int Lkv = cu_kv ? cu_kv[i + 1] - cu_kv[i] : L;   // rows of the segment's K/V
    int kv = kv_len ? kv_len[i] : Lkv;
    if (L < 0 || cu[i] < 0 || cu[i + 1] > T_cap || kv > Lkv || (L > 0 && kv <= 0)) {
      record_error(err, kErrLayout);
      kv = 0;
    }
    ntile[i] = (kv > 0) ? (L + kAttnRows * kAttnTiles - 1) / (kAttnRows * kAttnTiles) : 0;   // work units (tile groups) per head
    kvs[i] = kv;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < B; i += blockDim.x) {
    int rk = 0;
    for (int k = 0; k < B; ++k) rk += (kvs[k] > kvs[i]) || (kvs[k] == kvs[i] && k < i);
    rank[i] = rk;
  }
  __syncthreads();
  // offsets in rank order: a segment's units follow those of every segment
  // ranked before it (the ranks are a permutation of 0..B-1)
  for (int i = threadIdx.x; i < B; i += blockDim.x) {
    int before = 0;
    for (int k = 0; k < B; ++k) before += rank[k] < rank[i] ? ntile[k] : 0;
    off[i] = H * before;
  }
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int i = 0; i < B; ++i) acc += H * ntile[i];
    if (acc > max_units) {
      record_error(err, kErrCapacity);
      acc = max_units;
    }
    work_count[0] = acc;
    work_count[1] = 0;            // next unit handed out by the attention kernel
  }
  __syncthreads();
  for (int i = 0; i < B; ++i) {
    const int n = H * ntile[i];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const int idx = off[i] + k;
      if (idx < max_units) {
        const int g = k % ntile[i];
        const int tiles = (cu[i + 1] - cu[i] + kAttnRows - 1) / kAttnRows;
        work[idx] = make_int4(i, k / ntile[i], g * kAttnTiles, min(kAttnTiles, tiles - g * kAttnTiles));
      }
    }
  }
}

}  // namespace seer
