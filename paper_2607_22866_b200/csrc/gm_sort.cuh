// One-warp sort of packed (column, position) keys in registers and the summation of runs of equal columns: used for the
// small chunks of heavy rows and for light rows.
#pragma once
#include "gm_common.cuh"

namespace gm {

// Sorts 32 * K packed keys, K per lane, element e = r * 32 + lane in key[r]; ascending in e afterwards.
// Steps whose partner sits in another lane are the same instruction sequence for every step width, so they run
// as loops over the width; only the steps that pair registers are unrolled.  (Fully unrolled, the networks of
// all K together did not fit the instruction cache, and the warps of a block run different K.)
template <typename Key, int K>
__device__ __forceinline__ void warp_sort_keys(Key (&key)[K], int lane) {
  auto lane_step = [&](int mask, bool lower) {  // partner: same register, lane ^ mask; the lower lane keeps the smaller key
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const Key o = __shfl_xor_sync(0xffffffffu, key[r], mask);
      key[r] = lower ? min(key[r], o) : max(key[r], o);
    }
  };
  // merges inside one register row (k = 2 .. 32): first step partner e ^ (k - 1), then e ^ j for j = k/4 .. 1
#pragma unroll 1
  for (int k = 2; k <= 32; k <<= 1) {
    lane_step(k - 1, (lane & (k >> 1)) == 0);
#pragma unroll 1
    for (int j = k >> 2; j > 0; j >>= 1) lane_step(j, (lane & j) == 0);
  }
  // merges across register rows (k = 64 .. 32 K)
#pragma unroll
  for (int k = 64; k <= 32 * K; k <<= 1) {
    const int rm = k / 32 - 1;  // first step: partner register r ^ rm, partner lane lane ^ 31
#pragma unroll
    for (int r = 0; r < K; ++r) {
      if ((r ^ rm) > r) {
        const Key a = key[r], b = key[r ^ rm];
        const Key oa = __shfl_xor_sync(0xffffffffu, b, 31);
        const Key ob = __shfl_xor_sync(0xffffffffu, a, 31);
        key[r] = min(a, oa);
        key[r ^ rm] = max(b, ob);
      }
    }
#pragma unroll
    for (int j = k >> 2; j >= 32; j >>= 1) {  // partner in the same lane
      const int rj = j / 32;
#pragma unroll
      for (int r = 0; r < K; ++r) {
        if ((r & rj) == 0) {
          const Key a = key[r], b = key[r | rj];
          key[r] = min(a, b);
          key[r | rj] = max(a, b);
        }
      }
    }
#pragma unroll 1
    for (int j = 16; j > 0; j >>= 1) lane_step(j, (lane & j) == 0);
  }
}

// Sorted keys (n valid ones) -> entries: the lane that owns a run's first element adds the run up in the order of the
// positions (the low BITS bits of a key, indices into s_val) and writes it; returns the number of runs.
// s_key: 32 * K entries of this warp's shared memory.
template <typename V, typename Key, int K, int BITS>
__device__ __forceinline__ int warp_sum_runs(const Key (&key)[K], int n, Key* s_key, const V* s_val, u32 col_base, int32_t* col, V* val) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < K; ++r) s_key[r * 32 + lane] = key[r];
  __syncwarp();
  int base = 0;
#pragma unroll
  for (int r = 0; r < K; ++r) {
    if (r * 32 < n) {  // warp-uniform
      const int e = r * 32 + lane;
      const Key c = key[r] >> BITS;
      const bool head = e < n && (e == 0 || (s_key[e - 1] >> BITS) != c);
      const u32 heads = __ballot_sync(0xffffffffu, head);
      if (head) {
        V sum = s_val[static_cast<u32>(key[r]) & ((1u << BITS) - 1u)];
        for (int q = e + 1; q < n; ++q) {
          const Key kq = s_key[q];
          if ((kq >> BITS) != c) break;
          sum += s_val[static_cast<u32>(kq) & ((1u << BITS) - 1u)];
        }
        const int p = base + __popc(heads & lanemask_lt());
        col[p] = static_cast<int32_t>(col_base + static_cast<u32>(c));
        val[p] = sum;
      }
      base += __popc(heads);
    }
  }
  return base;
}

}  // namespace gm
