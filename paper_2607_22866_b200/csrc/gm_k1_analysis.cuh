// K1 — row analysis (InterOffsets and ThreshPartition of Algorithm 3, Section III-A).
//   IP_i = sum over stored entries j of A[i,:] of nnz(B[A.col[j], :])
//   heavy iff IP_i > tau; light rows are listed by the kernel that will take them.
// One launch does all of it for a whole matrix: products per row, the classes, the room every light row gets in the
// light rows' staging area, the totals the host needs (written straight into page-locked host memory by the last block
// to finish) and, per tile of rows, what the heavy rows' lists need.  A second launch (only when there are heavy rows)
// turns the tile sums into the heavy rows' lists.
// What bounds it: the dependent chain row_ptr -> column of A -> row_ptr of B on small inputs, the gather of B's row_ptr
// on large ones.  Before, the same facts took nine launches (products per entry, a prefix sum over the entries, row
// differences, binning and a second prefix sum): 24.6 us back to back for the row sums of R-MAT scale 15, and 175 us of
// kernels for a 1024^2 5-point grid.
// For the paths that expand products in a flattened space it also lays out a segment table: one segment per stored
// entry of a heavy row (a whole row of B scaled by one value of A), in row order, so that heavy row h owns the
// contiguous product range [heavy_base[h], heavy_base[h+1]).
#pragma once
#include "gm_common.cuh"

namespace gm {

// Classes of rows.  0: merged by one thread (few short rows of B); 1..6: sorted by one warp, at most 32 << (class - 1)
// products; 7..: hash accumulator, class c at most hash_cap[c - 7] products.
constexpr int kMergeClass = 0;
constexpr int kSortClass0 = 1;
constexpr int kSortClasses = 6;
constexpr int kHashClass0 = kSortClass0 + kSortClasses;
constexpr int kMaxHashClasses = 8;
constexpr int kRowClasses = kHashClass0 + kMaxHashClasses;
// A merged row has at most this many entries in A and products.  Product calls, us, merged / sorted: 5-point grids of 1024^2 points fp64
// 254 / 936, of 256^2 90 / 130; 262144 rows of scattered columns, 4 entries a row 195 / 257, 5 321 / 305, 6 420 / 378, 8 708 / 409: with
// more than four scattered lists the sort is the faster one, with lists that neighbouring rows share the merge stays ahead.
// Twice the products or the entries, sorted / merged: 8 x 12 552 / 1037, 12 x 8 564 / 1596.
constexpr int kMergeMaxLists = 8;
constexpr int kMergeMaxProducts = 64;
constexpr int kSortMaxProducts = 32 << (kSortClasses - 1);
// Below this many rows one thread per row leaves the device empty: scattered, 16384 rows, 5 entries a row 94 us sorted, 116 merged
// (2 entries 88 and 81, grids of 128^2 points 94 and 83).
constexpr i64 kMergeMinRows = 1 << 16;

struct RowRules {
  i64 tau, c_cols;
  int merge;                      // 1: rows that fit the merge kernel go there
  int sort_max;                   // rows of at most this many products are sorted by one warp (0: none)
  int n_hash;
  int hash_cap[kMaxHashClasses];
};

struct K1Totals {
  u64 products_total;
  u64 products_heavy;
  u64 products_max_row;
  u64 c_nnz_upper;
  u64 rows_heavy;
  u64 rows_empty;
  u64 nnz_a_heavy;
  u64 staged_light;               // products of the rows that are merged or sorted: room in the light staging area
  u64 merge_max_lists;            // most entries of A in a merged row
  u64 class_rows[kRowClasses];
  u64 done;                       // blocks finished (the last one hands the totals to the host)
};
constexpr int kK1Words = sizeof(K1Totals) / 8;

constexpr int kHeavyRows = 1024;
struct HeavyTile {  // what kHeavyRows consecutive rows add to the heavy rows' lists
  u64 products;
  u32 rows, pad;
  u64 nnz_a;
};

// How the rows are cut.  Rows of a power-law matrix have one to tens of thousands of entries and the long ones are
// neighbours (128 rows of R-MAT scale 15 hold a ninth of all entries), so the blocks share out rows and entries together:
// think of the entries and the row ends as one sequence, row after row (row r starts at item row_ptr[r] + r), and give
// every block T consecutive items.  A row that lies in one tile is summed there; the (at most two) rows a tile shares
// with its neighbours are summed with atomics, and the last tile to add its part goes on with the row.
// (Row sums of R-MAT scale 15: 6.7 us this way, 47 with a warp's lanes over rows, 120 with tiles of 128 rows.)
constexpr int kK1Threads = 256;

constexpr int kK1Small = 512, kK1Large = 2048;
// Items per tile: a small matrix is cut finer, so that more SMs have a block.
inline int k1_tile_items(i64 n_rows, i64 nnz_a, int num_sms) { return n_rows + nnz_a <= static_cast<i64>(num_sms) * 1024 ? kK1Small : kK1Large; }

// Largest r in [0, n_rows] with row_ptr[r] + r <= d, by one warp: 32 probes a step.
__device__ __forceinline__ i64 find_row(const i64* __restrict__ row_ptr, i64 n_rows, i64 d) {
  const int lane = threadIdx.x & 31;
  i64 lo = 0, hi = min(n_rows, d);  // the answer is in [lo, hi]
  while (lo < hi) {
    const i64 step = (hi - lo + 31) / 32;
    const i64 r = lo + step * (lane + 1);
    const bool ok = r <= hi && row_ptr[r] + r <= d;
    const int k = __popc(__ballot_sync(0xffffffffu, ok));  // (monotone: the first k probes hold)
    lo += step * k;
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// P: type of a warp's prefix sums.  A warp has T / 8 entries of the tile, at most 256, so 32 bits do for what is before
// each of them when B has at most 2^24 columns; the warp's total, which can be 2^32 then, is kept in 64.
template <int T, typename P>
struct K1Tile {
  i64 r0, r1;  // row of the first item, and of the first item after the tile
  i64 e0;      // first entry
  int n_rows;  // row ends in the tile
  int n_entries;
  int off[T + 1];    // start of row r0 + i relative to e0 (i = 0: at least 0)
  P pre[T + 1];      // exclusive prefix sums of the products per entry, inside the warp that loaded it
  i64 base[kK1Threads / 32 + 1];  // products before each warp's first entry
  i64 sum[kK1Threads / 32];
  __device__ __forceinline__ i64 before(int q) const { return base[q / (T / (kK1Threads / 32))] + static_cast<i64>(pre[q]); }
};

// Rows at the first items of tiles `tile`, `tile` + stride, ... (kK1Ahead of them, as far as there are any) and behind their last, a warp
// each: s_row[2 k] and s_row[2 k + 1].  Ends with a barrier.
constexpr int kK1Ahead = kK1Threads / 64;  // tiles whose rows are looked up together
template <int T>
__device__ __forceinline__ void k1_find_rows(const i64* __restrict__ a_row_ptr, i64 n_rows, i64 nnz_a, i64 tile, i64 stride, i64 n_tiles, i64* s_row) {
  const int warp = threadIdx.x >> 5;
  const i64 t = tile + (warp >> 1) * stride;
  if (t < n_tiles) {
    const i64 r = find_row(a_row_ptr, n_rows, min((t + (warp & 1)) * T, n_rows + nnz_a));
    if ((threadIdx.x & 31) == 0) s_row[warp] = r;
  }
  __syncthreads();
}

// Loads the rows of a tile that begins in row r0 and ends in row r1, and the prefix sums of its entries' products.  Ends with a barrier.
template <int T, typename P>
__device__ __forceinline__ void k1_load_tile(K1Tile<T, P>& s, const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col,
                                             i64 n_rows, i64 nnz_a, const i64* __restrict__ b_row_ptr, i64 tile, i64 r0, i64 r1) {
  const int tid = threadIdx.x, warp = tid >> 5;
  const i64 d0 = tile * T, d1 = min(d0 + T, n_rows + nnz_a);
  const i64 e0 = d0 - r0;
  const int nr = static_cast<int>(r1 - r0), ne = static_cast<int>(d1 - r1 - e0);
  if (tid == 0) { s.r0 = r0; s.r1 = r1; s.e0 = e0; s.n_rows = nr; s.n_entries = ne; }
  // every warp takes a run of consecutive entries, 32 at a time
  constexpr int kPer = T / kK1Threads;
  const int lane = tid & 31, q0 = warp * (32 * kPer) + lane;
  int len[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int q = q0 + k * 32;
    len[k] = 0;
    if (q < ne) {
      const int32_t c = a_col[e0 + q];
      len[k] = static_cast<int>(b_row_ptr[c + 1] - b_row_ptr[c]);
    }
  }
  for (int i = tid; i <= nr; i += kK1Threads) s.off[i] = static_cast<int>(max(a_row_ptr[r0 + i] - e0, i64{0}));
  i64 run = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const P inc = warp_inclusive_scan(static_cast<P>(len[k]));
    s.pre[q0 + k * 32] = static_cast<P>(run) + inc - static_cast<P>(len[k]);
    run += static_cast<i64>(__shfl_sync(0xffffffffu, inc, 31));
  }
  if (lane == 0) s.sum[warp] = run;
  __syncthreads();
  if (tid <= kK1Threads / 32) {
    i64 base = 0;
    for (int w = 0; w < tid; ++w) base += s.sum[w];
    s.base[tid] = base;
    if (tid == 0) s.pre[T] = 0;  // (position T belongs to the warp after the last)
  }
  __syncthreads();
}

// Products of the tile's part of local row i (0 .. n_rows; the last one goes on in the next tile).
template <int T, typename P>
__device__ __forceinline__ i64 k1_part(const K1Tile<T, P>& s, int i) {
  return s.before(i < s.n_rows ? s.off[i + 1] : s.n_entries) - s.before(s.off[i]);
}
// Does the tile share local row i with other tiles, and does it hold any item of it?
template <int T, typename P>
__device__ __forceinline__ bool k1_shared_row(const K1Tile<T, P>& s, int i, const i64* __restrict__ a_row_ptr) {
  return i == s.n_rows || (i == 0 && a_row_ptr[s.r0] < s.e0);
}
template <int T, typename P>
__device__ __forceinline__ bool k1_touched(const K1Tile<T, P>& s, int i) {
  return i < s.n_rows || s.n_entries > s.off[i];
}

template <int T, typename P>
__global__ void __launch_bounds__(kK1Threads) k1_rows(
    const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col, i64 n_rows, i64 nnz_a, const i64* __restrict__ b_row_ptr,
    RowRules rules, i64* __restrict__ ip, u32* __restrict__ parts,  // zero-initialised: products; tiles that have added theirs
    int32_t* __restrict__ heavy_flag, int32_t* __restrict__ row_nnz,
    i64* __restrict__ light_off,              // per row: place in the light staging area, -1: none
    int32_t* __restrict__ rows_out, i64 list_stride,  // class c's rows at rows_out + c * list_stride
    HeavyTile* __restrict__ heavy_tiles,      // zero-initialised, per kHeavyRows rows
    K1Totals* __restrict__ totals, u64* __restrict__ host_totals) {
  __shared__ K1Tile<T, P> s;
  __shared__ u32 s_cls[T + 1];   // per row: class << 16 | rank in the tile's part of the class list
  __shared__ u32 s_room[T + 1];  // per row: place in the tile's part of the staging area
  __shared__ u32 s_cnt[kRowClasses], s_room_n;
  __shared__ u32 s_base[kRowClasses];
  __shared__ u64 s_stage_base;
  __shared__ u64 s_tot[8];
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 8) s_tot[tid] = 0;
  u64 tot = 0, hev = 0, hnz = 0, mx = 0, up = 0, ml = 0;
  u32 nh = 0, ne = 0;
  const i64 n_tiles = (n_rows + nnz_a + T - 1) / T;
  // (a few blocks per SM, each with many tiles: the totals sit in one line of L2, and a set of atomics per tile was most
  // of this kernel's time.  The blocks go round-robin over the tiles: with a run of neighbouring tiles for each, 1400 tiles kept 700 of 888
  // blocks busy, and the Zipf pair of 2^20 rows took 315 us here instead of 277.  The eight warps look up the rows of a block's next four
  // tiles together: with two warps that did so for every tile while the others waited, that pair took 290 us, the 1024^2 grid 55
  // instead of 50, ER of 200000 rows of 12 56 instead of 54.)
  __shared__ i64 s_row[2 * kK1Ahead];
  int ahead = 0;
  for (i64 tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ahead = (ahead + 1) % kK1Ahead) {
    if (tid < kRowClasses) s_cnt[tid] = 0;
    if (tid == 32) s_room_n = 0;
    if (ahead == 0) k1_find_rows<T>(a_row_ptr, n_rows, nnz_a, tile, gridDim.x, n_tiles, s_row);
    k1_load_tile<T, P>(s, a_row_ptr, a_col, n_rows, nnz_a, b_row_ptr, tile, s_row[2 * ahead], s_row[2 * ahead + 1]);
    for (int i0 = 0; i0 <= s.n_rows; i0 += kK1Threads) {
      // ---- one thread per row: class, room, totals
      const int i = i0 + tid;
      int cls = -1;
      i64 p = 0;
      bool mine = false, heavy = false;
      const i64 row = s.r0 + i;
      i64 entries = 0;
      if (i <= s.n_rows && row < n_rows && k1_touched<T, P>(s, i)) {
        p = k1_part<T, P>(s, i);
        const i64 first = a_row_ptr[row], end = a_row_ptr[row + 1];
        entries = end - first;
        mine = true;
        if (k1_shared_row<T, P>(s, i, a_row_ptr)) {
          const u32 tiles = static_cast<u32>((end + row) / T - (first + row) / T) + 1;
          if (tiles > 1) {
            if (p) atomicAdd(reinterpret_cast<u64*>(&ip[row]), static_cast<u64>(p));
            __threadfence();
            mine = atomicAdd(&parts[row], 1u) == tiles - 1;
            if (mine) {
              __threadfence();
              p = static_cast<i64>(atomicAdd(reinterpret_cast<u64*>(&ip[row]), 0ull));
            }
          } else {
            ip[row] = p;
          }
        } else {
          ip[row] = p;
        }
      }
      if (mine) {
        heavy = p > rules.tau;
        heavy_flag[row] = heavy ? 1 : 0;
        row_nnz[row] = 0;
        if (p == 0) {
          ++ne;
        } else if (!heavy) {
          if (rules.merge && entries <= kMergeMaxLists && p <= kMergeMaxProducts) {
            cls = kMergeClass;
            ml = static_cast<u64>(entries) > ml ? static_cast<u64>(entries) : ml;
          } else if (p <= rules.sort_max) {
            cls = kSortClass0;
            while (p > (32 << (cls - kSortClass0))) ++cls;
          } else {
            cls = kHashClass0;
            while (p > rules.hash_cap[cls - kHashClass0]) ++cls;
          }
        }
        tot += p;
        mx = static_cast<u64>(p) > mx ? static_cast<u64>(p) : mx;
        up += p < rules.c_cols ? p : rules.c_cols;
      }
      const u32 hm = __ballot_sync(0xffffffffu, heavy);
      if (heavy) {
        hev += p; hnz += entries; ++nh;
      }
      if (hm) {  // the heavy rows' facts per group of kHeavyRows rows: a warp's rows are nearly always in one group
        const i64 g = row / kHeavyRows;
        const i64 g0 = __shfl_sync(0xffffffffu, g, __ffs(hm) - 1);
        const bool same = __ballot_sync(0xffffffffu, heavy && g != g0) == 0;
        const u64 wp = warp_sum(heavy ? static_cast<u64>(p) : 0), wz = warp_sum(heavy ? static_cast<u64>(entries) : 0);
        if (same) {
          if (lane == 0) {
            atomicAdd(&heavy_tiles[g0].products, wp);
            atomicAdd(&heavy_tiles[g0].nnz_a, wz);
            atomicAdd(&heavy_tiles[g0].rows, static_cast<u32>(__popc(hm)));
          }
        } else if (heavy) {
          atomicAdd(&heavy_tiles[g].products, static_cast<u64>(p));
          atomicAdd(&heavy_tiles[g].nnz_a, static_cast<u64>(entries));
          atomicAdd(&heavy_tiles[g].rows, 1u);
        }
      }
      // ---- places inside the tile's share of the class lists and of the light staging area
      const bool staged = cls >= 0 && cls < kHashClass0;
      const u32 room = staged ? static_cast<u32>(p) : 0u;
      const u32 inc = warp_inclusive_scan(room);
      u32 at = 0;
      if (lane == 31 && inc) at = atomicAdd(&s_room_n, inc);
      at = __shfl_sync(0xffffffffu, at, 31) + inc - room;
      u32 cr = 0xffffffffu;
      for (u32 left = __reduce_or_sync(0xffffffffu, cls >= 0 ? 1u << cls : 0u); left; left &= left - 1) {  // classes in this warp
        const int c = __ffs(left) - 1;
        const u32 m = __ballot_sync(0xffffffffu, cls == c);
        u32 base = 0;
        if (lane == 0) base = atomicAdd(&s_cnt[c], static_cast<u32>(__popc(m)));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (cls == c) cr = (static_cast<u32>(c) << 16) | (base + __popc(m & lanemask_lt()));
      }
      if (i <= s.n_rows) {
        s_cls[i] = mine ? (cls >= 0 ? cr : 0xffff0000u) : 0xffffffffu;
        s_room[i] = staged ? at : 0xffffffffu;
      }
    }
    __syncthreads();
    if (tid < kRowClasses) s_base[tid] = s_cnt[tid] ? static_cast<u32>(atomicAdd(&totals->class_rows[tid], static_cast<u64>(s_cnt[tid]))) : 0;
    else if (tid == 32) s_stage_base = s_room_n ? atomicAdd(&totals->staged_light, static_cast<u64>(s_room_n)) : 0;
    __syncthreads();
    for (int i = tid; i <= s.n_rows; i += kK1Threads) {
      const u32 cr = s_cls[i];
      if (cr == 0xffffffffu) continue;  // another tile's row
      const i64 row = s.r0 + i;
      light_off[row] = s_room[i] == 0xffffffffu ? -1 : static_cast<i64>(s_stage_base) + s_room[i];
      const u32 cls = cr >> 16;
      if (cls < kRowClasses) rows_out[static_cast<i64>(cls) * list_stride + s_base[cls] + (cr & 0xffffu)] = static_cast<int32_t>(row);
    }
    __syncthreads();  // the shared arrays are reused by the next tile
  }
  tot = warp_sum(tot); up = warp_sum(up); ne = warp_sum(ne);
  hev = warp_sum(hev); hnz = warp_sum(hnz); nh = warp_sum(nh);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u64 m2 = __shfl_xor_sync(0xffffffffu, mx, o), l2 = __shfl_xor_sync(0xffffffffu, ml, o);
    mx = m2 > mx ? m2 : mx;
    ml = l2 > ml ? l2 : ml;
  }
  if (lane == 0) {
    if (tot) { atomicAdd(&s_tot[0], tot); atomicAdd(&s_tot[1], up); atomicMax(&s_tot[2], mx); atomicMax(&s_tot[3], ml); }
    if (ne) atomicAdd(&s_tot[4], static_cast<u64>(ne));
    if (nh) { atomicAdd(&s_tot[5], hev); atomicAdd(&s_tot[6], hnz); atomicAdd(&s_tot[7], static_cast<u64>(nh)); }
  }
  __syncthreads();
  if (tid < 8 && s_tot[tid]) {
    u64* const where[8] = {&totals->products_total, &totals->c_nnz_upper, &totals->products_max_row, &totals->merge_max_lists,
                           &totals->rows_empty, &totals->products_heavy, &totals->nnz_a_heavy, &totals->rows_heavy};
    if (tid == 2 || tid == 3) atomicMax(where[tid], s_tot[tid]);
    else atomicAdd(where[tid], s_tot[tid]);
  }
  if (warp == 0) {
    __threadfence();
    __syncwarp();
    if (tid == 0) s_last = atomicAdd(&totals->done, 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    const volatile u64* src = reinterpret_cast<const volatile u64*>(totals);
    for (int w = tid; w < kK1Words; w += kK1Threads) host_totals[w] = src[w];  // (the host reads after a synchronisation)
  }
}

// Products per row alone, for callers that keep no plan (see gm_row_products_noalloc): ip is zero-initialised.
template <int T, typename P>
__global__ void __launch_bounds__(kK1Threads) k1_row_products_only(const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col,
                                                                   i64 n_rows, i64 nnz_a, const i64* __restrict__ b_row_ptr,
                                                                   i64* __restrict__ ip) {
  __shared__ K1Tile<T, P> s;
  __shared__ i64 s_row[2];  // (a block has one tile)
  k1_find_rows<T>(a_row_ptr, n_rows, nnz_a, blockIdx.x, gridDim.x, gridDim.x, s_row);
  k1_load_tile<T, P>(s, a_row_ptr, a_col, n_rows, nnz_a, b_row_ptr, blockIdx.x, s_row[0], s_row[1]);
  for (int i = threadIdx.x; i <= s.n_rows; i += kK1Threads) {
    const i64 row = s.r0 + i;
    if (row >= n_rows || !k1_touched<T, P>(s, i)) continue;
    const i64 p = k1_part<T, P>(s, i);
    if (!k1_shared_row<T, P>(s, i, a_row_ptr)) ip[row] = p;
    else if (p) atomicAdd(reinterpret_cast<u64*>(&ip[row]), static_cast<u64>(p));
  }
}

// Heavy rows in row order: x_heavy[h] = row, heavy_base / heavy_nz_off = exclusive prefix sums of their products and
// entries.  One block per kHeavyRows rows; it adds up the groups before its own (a few thousand at most) by itself, so
// there is no separate pass for the prefix.
constexpr int kHeavyThreads = 256;
static_assert(kHeavyRows == 4 * kHeavyThreads, "four rows per thread");
__global__ void __launch_bounds__(kHeavyThreads) k1_heavy_lists(const i64* __restrict__ ip, const int32_t* __restrict__ heavy_flag,
                                                                const i64* __restrict__ a_row_ptr, i64 n_rows,
                                                                const HeavyTile* __restrict__ tiles, int32_t* __restrict__ x_heavy,
                                                                i64* __restrict__ heavy_base, i64* __restrict__ heavy_nz_off) {
  __shared__ i64 s_tmp[3][33];
  const i64 r0 = static_cast<i64>(blockIdx.x) * kHeavyRows;
  i64 b_rows = 0, b_prod = 0, b_nnz = 0;
  for (i64 t = threadIdx.x; t < static_cast<i64>(blockIdx.x); t += kHeavyThreads) {
    const HeavyTile h = tiles[t];
    b_rows += h.rows; b_prod += static_cast<i64>(h.products); b_nnz += static_cast<i64>(h.nnz_a);
  }
  const i64 i0 = r0 + threadIdx.x * 4;
  bool heavy[4];
  i64 p[4], z[4];
  i64 m_rows = 0, m_prod = 0, m_nnz = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const i64 i = i0 + k;
    heavy[k] = i < n_rows && heavy_flag[i];
    p[k] = heavy[k] ? ip[i] : 0;
    z[k] = heavy[k] ? a_row_ptr[i + 1] - a_row_ptr[i] : 0;
    m_rows += heavy[k]; m_prod += p[k]; m_nnz += z[k];
  }
  // prefix over the block's threads, and the groups before the block (every thread holds a part of those)
  i64 t_rows, t_prod, t_nnz, g_rows, g_prod, g_nnz;
  i64 e_rows = block_exclusive_scan(m_rows, s_tmp[0], &t_rows);
  i64 e_prod = block_exclusive_scan(m_prod, s_tmp[1], &t_prod);
  i64 e_nnz = block_exclusive_scan(m_nnz, s_tmp[2], &t_nnz);
  __syncthreads();
  block_exclusive_scan(b_rows, s_tmp[0], &g_rows);
  block_exclusive_scan(b_prod, s_tmp[1], &g_prod);
  block_exclusive_scan(b_nnz, s_tmp[2], &g_nnz);
  e_rows += g_rows; e_prod += g_prod; e_nnz += g_nnz;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (heavy[k]) {
      x_heavy[e_rows] = static_cast<int32_t>(i0 + k);
      heavy_base[e_rows] = e_prod;
      heavy_nz_off[e_rows] = e_nnz;
      ++e_rows; e_prod += p[k]; e_nnz += z[k];
    }
  }
  if (r0 + kHeavyRows >= n_rows && threadIdx.x == 0) {
    heavy_base[g_rows + t_rows] = g_prod + t_prod;
    heavy_nz_off[g_rows + t_rows] = g_nnz + t_nnz;
  }
}

// Segment s (the s-th stored entry of the heavy rows, in row order) copies B's entries from position seg_bstart[s], is
// scaled by A.val[seg_j[s]] and has seg_len[s] products (their prefix sum is seg_off).
constexpr int kSegRun = 256;
__global__ void k1_heavy_segments(const int32_t* __restrict__ x_heavy, i64 n_heavy, const i64* __restrict__ heavy_nz_off,
                                  const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col,
                                  const i64* __restrict__ b_row_ptr, i64 n_seg, int32_t* __restrict__ seg_len,
                                  i64* __restrict__ seg_bstart, i64* __restrict__ seg_j,
                                  int32_t* __restrict__ seg_brow, int32_t* __restrict__ seg_hrow) {
  // A warp takes kSegRun consecutive segments: one search for its first, then a step forward where a row ends.  (A search
  // per segment took 184 us for the 11.5 M segments of the clipped-Zipf pair.)
  const int lane = threadIdx.x & 31;
  const i64 s0 = (static_cast<i64>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kSegRun;
  if (s0 >= n_seg) return;
  i64 h = 0;
  for (i64 hi = n_heavy - 1; h < hi;) {  // last row that starts at or before s0 (rows with no entries are never heavy)
    const i64 step = (hi - h + 31) / 32;
    const i64 r = h + step * (lane + 1);
    const int ok = __popc(__ballot_sync(0xffffffffu, r <= hi && heavy_nz_off[r] <= s0));
    h += step * ok;
    hi = min(hi, h + step - 1);
  }
  const i64 s1 = min(n_seg, s0 + kSegRun);
  for (i64 s = s0 + lane; s < s1; s += 32) {
    while (heavy_nz_off[h + 1] <= s) ++h;
    const i64 j = a_row_ptr[x_heavy[h]] + (s - heavy_nz_off[h]);
    const int32_t k = a_col[j];
    const i64 b0 = b_row_ptr[k];
    seg_len[s] = static_cast<int32_t>(b_row_ptr[k + 1] - b0);
    seg_bstart[s] = b0;
    seg_j[s] = j;
    seg_brow[s] = k;
    seg_hrow[s] = static_cast<int32_t>(h);
  }
}

// Lists rows [row0, row0 + n_rows) of the hash classes again by their entry counts, for the numeric pass: bin b holds
// rows with cap[b - 1] < entries <= cap[b].  Rows that are not in a hash class (light_off >= 0: staged; heavy; empty)
// are left out.
constexpr int kMaxLightBins = 8;
static_assert(kMaxLightBins <= kMaxHashClasses, "the bins serve as classes when every light row is hashed");
struct LightBins {
  int n_bins;
  int cap[kMaxLightBins];
};
__global__ void __launch_bounds__(256) k1_bin_rows(const int32_t* __restrict__ size, const int32_t* __restrict__ heavy_flag,
                                                   const i64* __restrict__ light_off, i64 row0, i64 n_rows, LightBins lb,
                                                   i64 bin_stride, int* __restrict__ bin_fill, int32_t* __restrict__ rows_out) {
  __shared__ int s_cnt[8][kMaxLightBins];
  __shared__ int s_base[kMaxLightBins];
  const i64 i = row0 + static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x;
  int bin = -1, rank = 0;
  if (i < row0 + n_rows && !heavy_flag[i] && light_off[i] < 0) {
    const int sz = size[i];
    if (sz > 0) {
      bin = 0;
      while (bin < lb.n_bins - 1 && sz > lb.cap[bin]) ++bin;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int b = 0; b < lb.n_bins; ++b) {
    const u32 m = __ballot_sync(0xffffffffu, bin == b);
    if (bin == b) rank = __popc(m & lanemask_lt());
    if (lane == 0) s_cnt[warp][b] = __popc(m);
  }
  __syncthreads();
  if (static_cast<int>(threadIdx.x) < lb.n_bins) {
    int run = 0;
    for (int w = 0; w < 8; ++w) { const int c = s_cnt[w][threadIdx.x]; s_cnt[w][threadIdx.x] = run; run += c; }
    s_base[threadIdx.x] = run ? atomicAdd(&bin_fill[threadIdx.x], run) : 0;
  }
  __syncthreads();
  if (bin >= 0) rows_out[bin * bin_stride + s_base[bin] + s_cnt[warp][bin] + rank] = static_cast<int32_t>(i);
}

}  // namespace gm
