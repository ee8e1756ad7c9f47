// One-warp sort of packed (column, position) keys in registers and the summation of runs of equal columns: used for the
// small chunks of heavy rows and for light rows.
#pragma once
#include "gm_common.cuh"

namespace gm {

// Sorts 32 * K packed keys, K per lane, ascending; element e = lane * K + r ends in key[r] (a bitonic network whose merges
// begin with the mirrored partner, so that every run is ascending).
// A lane's elements are neighbours, so that the short strides, which every merge ends with, stay inside the lane: 15 of the 36
// steps for 256 keys exchange with another lane, against 33 with element r * 32 + lane in key[r], and an exchange takes a
// shuffle per key, of which an SM does one at a time.  (ER, 30011 rows of 144 products fp64:
// 75 -> 62 us; the sorts of the Zipf pair with 64-bit keys, rows up to 1024 products: the whole product 5.42 -> 4.95 ms.)
// The merges across lanes are the same instruction sequence for every width and run as a loop; only the steps inside a lane
// are unrolled.  (Fully unrolled, the networks of all K together did not fit the instruction cache, and the warps of a block
// run different K.)
// K: a power of two, or 3, 5, 6: the exchanges between lanes do not care, and inside a lane the smallest networks for so few are no longer
// than the strides for eight.  (Rows of 144 products padded to 160 instead of 256: 62 -> 55 us for ER of 30011 rows fp64; of 200000 rows fp32
// the call 563 -> 515.)
template <typename Key, int K>
__device__ __forceinline__ void warp_sort_keys(Key (&key)[K], int lane) {
  constexpr bool kPow2 = (K & (K - 1)) == 0;
  auto order = [](Key& a, Key& b) {
    const Key lo = min(a, b);
    b = max(a, b);
    a = lo;
  };
  auto network = [&]() {  // any order -> ascending, for the K that are no power of two (optimal networks, Knuth vol. 3, 5.3.4)
    auto o = [&](int i, int j) { order(key[i], key[j]); };
    if constexpr (K == 3) { o(0, 2); o(0, 1); o(1, 2); }
    if constexpr (K == 5) { o(0, 3); o(1, 4); o(0, 2); o(1, 3); o(0, 1); o(2, 4); o(1, 2); o(3, 4); o(2, 3); }
    if constexpr (K == 6) { o(0, 5); o(1, 3); o(2, 4); o(1, 2); o(3, 4); o(0, 3); o(2, 5); o(0, 1); o(2, 3); o(4, 5); o(1, 2); o(3, 4); }
    static_assert(kPow2 || K == 3 || K == 5 || K == 6, "no network");
  };
  auto strides_in_lane = [&](int from) {  // partner e ^ j for j = from .. 1
#pragma unroll
    for (int j = K / 2; j > 0; j >>= 1) {
      if (j > from) continue;
#pragma unroll
      for (int r = 0; r < K; ++r)
        if ((r & j) == 0) order(key[r], key[r | j]);
    }
  };
  // runs of K in every lane
  if constexpr (!kPow2) network();
  else {
#pragma unroll
    for (int k = 2; k <= K; k <<= 1) {
#pragma unroll
      for (int r = 0; r < K; ++r)
        if ((r ^ (k - 1)) > r) order(key[r], key[r ^ (k - 1)]);
      strides_in_lane(k / 4);
    }
  }
  // merges of the runs of w lanes with their neighbours'; the lower lane of a pair keeps the smaller keys
#pragma unroll 1
  for (int w = 1; w < 32; w <<= 1) {
    const bool lower = (lane & w) == 0;
    const int mask = 2 * w - 1;
#pragma unroll
    for (int r = 0; r < (K + 1) / 2; ++r) {  // mirrored: register K - 1 - r of lane ^ mask
      const Key a = key[r], b = key[K - 1 - r];
      const Key oa = __shfl_xor_sync(0xffffffffu, b, mask);
      key[r] = lower ? min(a, oa) : max(a, oa);
      if (r != K - 1 - r) {
        const Key ob = __shfl_xor_sync(0xffffffffu, a, mask);
        key[K - 1 - r] = lower ? min(b, ob) : max(b, ob);
      }
    }
#pragma unroll 1
    for (int j = w >> 1; j > 0; j >>= 1) {
      const bool first = (lane & j) == 0;
#pragma unroll
      for (int r = 0; r < K; ++r) {
        const Key o = __shfl_xor_sync(0xffffffffu, key[r], j);
        key[r] = first ? min(key[r], o) : max(key[r], o);
      }
    }
    if constexpr (kPow2) strides_in_lane(K / 2);
    else network();
  }
}

// Sorted keys (n valid ones) -> entries: the lane that owns a run's first element adds the run up in the order of the
// positions (the low BITS bits of a key, indices into s_val) and writes it; returns the number of runs.
// s_key: 32 * K entries of this warp's shared memory, 16-byte aligned.
template <typename V, typename Key, int K, int BITS>
__device__ __forceinline__ int warp_sum_runs(const Key (&key)[K], int n, Key* s_key, const V* s_val, u32 col_base, int32_t* col, V* val) {
  const int lane = threadIdx.x & 31;
  constexpr int kVec = 16 / sizeof(Key);
  if constexpr (K % kVec == 0) {
#pragma unroll
    for (int r = 0; r < K; r += kVec) {
      if constexpr (sizeof(Key) == 4) *reinterpret_cast<uint4*>(s_key + lane * K + r) = make_uint4(key[r], key[r + 1], key[r + 2], key[r + 3]);
      else *reinterpret_cast<ulonglong2*>(s_key + lane * K + r) = make_ulonglong2(key[r], key[r + 1]);
    }
  } else {
#pragma unroll
    for (int r = 0; r < K; ++r) s_key[lane * K + r] = key[r];
  }
  __syncwarp();
  int base = 0;
#pragma unroll
  for (int r = 0; r < K; ++r) {
    if (r * 32 < n) {  // warp-uniform
      const int e = r * 32 + lane;
      const Key k = s_key[e];
      const Key c = k >> BITS;
      const bool head = e < n && (e == 0 || (s_key[e - 1] >> BITS) != c);
      const u32 heads = __ballot_sync(0xffffffffu, head);
      if (head) {
        V sum = s_val[static_cast<u32>(k) & ((1u << BITS) - 1u)];
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
