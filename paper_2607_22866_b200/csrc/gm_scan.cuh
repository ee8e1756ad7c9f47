// Device-wide exclusive prefix sum without any wait between blocks.  Used for every row_ptr-like array on the path
// (C^.rowPtr, C^_reord.rowPtr, C.rowPtr of Algorithm 3).
//   up to one tile      one launch, one block
//   up to kScanSelfTiles two launches: tile sums, then every block adds up the sums of the tiles before its own itself
//                       (a few kilobytes out of L2) instead of waiting for a pass over them: the launch and its gap
//                       cost more than the re-reading
//   more                three launches, the middle one a single block over the tile sums
#pragma once
#include "gm_common.cuh"

namespace gm {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;  // 4096
constexpr i64 kScanSelfTiles = 2048;

inline i64 scan_tmp_elems(i64 n) { return (n + kScanTile - 1) / kScanTile + 2; }

// tile_sum[0] = carry, tile_sum[1 + t] = sum of tile t
template <typename In>
__global__ void __launch_bounds__(kScanThreads) scan_tile_sums(const In* __restrict__ in, i64 n, const i64* __restrict__ carry_in,
                                                              i64* __restrict__ tile_sum) {
  __shared__ i64 tmp[kScanThreads / 32];
  const i64 t0 = static_cast<i64>(blockIdx.x) * kScanTile;
  i64 s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const i64 i = t0 + k * kScanThreads + threadIdx.x;
    if (i < n) s += static_cast<i64>(in[i]);
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) tmp[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kScanThreads / 32; ++w) s += tmp[w];
    tile_sum[1 + blockIdx.x] = s;
    if (blockIdx.x == 0) tile_sum[0] = carry_in ? *carry_in : 0;
  }
}

// One block: tile_sum[0 .. n_tiles] -> inclusive prefixes (tile_sum[t] becomes the base of tile t).
__global__ void __launch_bounds__(1024) scan_spine(i64* __restrict__ tile_sum, i64 n_tiles) {
  __shared__ i64 tmp[33];
  i64 running = 0;
  for (i64 b = 0; b < n_tiles + 1; b += blockDim.x) {
    const i64 i = b + threadIdx.x;
    const i64 v = i < n_tiles + 1 ? tile_sum[i] : 0;
    i64 total;
    const i64 ex = block_exclusive_scan(v, tmp, &total);
    if (i < n_tiles + 1) tile_sum[i] = running + ex + v;
    running += total;
    __syncthreads();
  }
}

// MODE 0: tile_sum holds sums, the block adds up its own base; 1: it holds the bases (scan_spine ran); 2: one tile, no sums
template <typename In, typename Out, int MODE>
__global__ void __launch_bounds__(kScanThreads) scan_tiles(const In* __restrict__ in, i64 n, const i64* __restrict__ tile_sum,
                                                          const i64* carry_in, i64* carry_out, i64* host_total,
                                                          Out* __restrict__ out, Out* __restrict__ out2) {
  __shared__ i64 tmp[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  i64 base = 0;
  if constexpr (MODE == 0) {
    i64 s = 0;
    for (i64 t = threadIdx.x; t <= static_cast<i64>(blockIdx.x); t += kScanThreads) s += tile_sum[t];
    block_exclusive_scan(s, tmp, &base);
    __syncthreads();
  } else if constexpr (MODE == 1) {
    base = tile_sum[blockIdx.x];
  } else {
    base = carry_in ? *carry_in : 0;
  }
  // a warp owns 256 consecutive items, taken 32 at a time: coalesced, and the prefix inside the warp is running
  const i64 w0 = static_cast<i64>(blockIdx.x) * kScanTile + warp * (32 * kScanItems);
  i64 v[kScanItems];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const i64 i = w0 + k * 32 + lane;
    v[k] = i < n ? static_cast<i64>(in[i]) : 0;
  }
  i64 run = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const i64 inc = warp_inclusive_scan(v[k]);
    const i64 sum = __shfl_sync(0xffffffffu, inc, 31);
    v[k] = run + inc - v[k];
    run += sum;
  }
  i64 total;
  // (every lane contributes the warp's sum once: lane 31 of each warp)
  const i64 ex = block_exclusive_scan(lane == 0 ? run : i64{0}, tmp, &total);
  const i64 wbase = base + __shfl_sync(0xffffffffu, ex, 0);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const i64 i = w0 + k * 32 + lane;
    if (i < n) {
      out[i] = static_cast<Out>(wbase + v[k]);
      if (out2) out2[i] = static_cast<Out>(wbase + v[k]);
    }
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    out[n] = static_cast<Out>(base + total);
    if (carry_out) *carry_out = base + total;
    if (host_total) *host_total = base + total;  // (the host reads after a synchronisation)
  }
}

// out[0..n) = carry + exclusive prefix sums of in, out[n] = carry + total (out has n + 1 entries).
// out2 (optional, n entries) receives a second copy of out[0..n).  tmp has scan_tmp_elems(n) entries.  carry_in and
// carry_out (device, optional) may be the same address.  host_total (optional): page-locked host memory that also
// receives the total.  Returns the number of launches.
template <typename In, typename Out>
int exclusive_scan(const In* in, Out* out, i64 n, i64* tmp, const i64* carry_in, i64* carry_out, Out* out2, cudaStream_t st,
                   i64* host_total = nullptr) {
  static_assert(sizeof(Out) == 8, "offsets are 64-bit");
  const i64 tiles = (n + kScanTile - 1) / kScanTile;
  if (tiles <= 1) {
    scan_tiles<In, Out, 2><<<1, kScanThreads, 0, st>>>(in, n, nullptr, carry_in, carry_out, host_total, out, out2);
    return 1;
  }
  scan_tile_sums<In><<<static_cast<unsigned>(tiles), kScanThreads, 0, st>>>(in, n, carry_in, tmp);
  if (tiles <= kScanSelfTiles) {
    scan_tiles<In, Out, 0><<<static_cast<unsigned>(tiles), kScanThreads, 0, st>>>(in, n, tmp, nullptr, carry_out, host_total, out, out2);
    return 2;
  }
  scan_spine<<<1, 1024, 0, st>>>(tmp, tiles);
  scan_tiles<In, Out, 1><<<static_cast<unsigned>(tiles), kScanThreads, 0, st>>>(in, n, tmp, nullptr, carry_out, host_total, out, out2);
  return 3;
}

}  // namespace gm
