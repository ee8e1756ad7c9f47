// K6t — heavy rows without a staged intermediate matrix: the products of a row of C inside a range of columns are
// generated where they are summed.
//
// A row of B has ascending columns, so its entries inside any range of columns are one contiguous piece, and a table of
// boundaries per row of B (every `granule` columns) gives the piece of every range that starts and ends on a boundary.
// A *task* is one heavy row times one range of columns; a kernel that sums a task walks the row's entries of A, takes the
// piece of each row of B and scales it.  Against writing every product to a staging buffer and reading it back (K4, K5)
// that leaves out (4 + s_v) bytes written and read per product; B, which is what is read instead, mostly stays in L2.
//
// Ranges are chosen per row (k_task_count / k_task_emit) from its products per granule: as many neighbouring granules as
// one team can sum together.
//   small  at most small_max products, any width: sorted by one warp
//   mid    at most mid_max products, at most mid_width columns: a 128-thread block, symbolic then numeric pass
//   big    one granule, or part of one: dense accumulator; three blocks per SM, so that one block's flush runs next to the
//          others' sums
// A granule with very many products (a hub row's) is cut further into sub-ranges with about equally many products, so that
// no block is left alone with it at the end; the boundaries inside a row of B are then found by binary search.
// Results go to the staging area at the place of the task's products (sub-ranges: at the distance of their first column,
// there are more products than columns), from where the gather moves them once the entries are counted.
#pragma once
#include "gm_common.cuh"
#include "gm_k6_accumulate.cuh"
#include "gm_sort.cuh"

namespace gm {

struct __align__(16) HeavyTask {
  i64 a0;       // first entry of the row in A
  i64 off;      // place in the staging area (batch-relative)
  u32 n_a;      // entries of the row in A
  u32 lo, hi;   // columns [lo, hi)
  u32 n;        // products (0: a sub-range, not counted)
};
static_assert(sizeof(HeavyTask) == 32, "two 16-byte loads");

struct TaskRules {
  int granules;    // per row
  int log2_g;      // columns per granule
  int small_max, mid_max;
  u32 mid_width, small_width;
  u32 split_above; // products of one granule above which it is cut
  int max_parts;   // ... into at most this many sub-ranges (a power of two)
};
constexpr int kMaxParts = 16;

// Counts about panels (see gm_k6_panels.cuh).  Entries of A in all that were found; blocks of k_panel_cut that are through; unordered: a
// row of B does not ascend.  Of the rows that k_panel_similar looked at closer: columns tried and found in the row before, rows of B, their
// pieces and entries.  Gain: what the panels are expected to save, in products.
enum PanelCount { kPanelsFound = 0, kPanelUnits, kPanelEntries, kPanelBlocks, kPanelUnordered, kPanelTried, kPanelHits, kPanelSampled, kPanelPieces, kPanelSampleLen, kPanelGain, kPanelCounts };

// bound[k * (granules + 1) + c] = position in B's arrays of the first entry of row k with column >= c << log2_g.
// A thread per boundary, each a binary search inside the row.
// longest: (entries << 32) | row of the longest row of B.
__global__ void __launch_bounds__(256) k_piece_bounds(const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, i64 n_rows_b,
                                                      int granules, int log2_g, u32* __restrict__ bound, u64* __restrict__ longest) {
  const i64 per_row = granules + 1;
  const i64 n = n_rows_b * per_row;
  u64 best = 0;
  for (i64 i = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += static_cast<i64>(gridDim.x) * blockDim.x) {
    const i64 k = i / per_row;
    const i64 c = i - k * per_row;
    const i64 rs = b_row_ptr[k], re = b_row_ptr[k + 1];
    i64 lo = rs, hi = re;
    if (c == 0) {
      hi = rs;
      const u64 len = static_cast<u64>(re - rs) << 32 | static_cast<u64>(k);
      best = len > best ? len : best;
    } else if (c == granules) {
      lo = re;
    }
    while (lo < hi) {
      const i64 mid = (lo + hi) >> 1;
      if ((static_cast<i64>(b_col[mid]) >> log2_g) >= c) hi = mid; else lo = mid + 1;
    }
    bound[i] = static_cast<u32>(lo);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { const u64 x = __shfl_xor_sync(0xffffffffu, best, o); best = x > best ? x : best; }
  if ((threadIdx.x & 31) == 0 && best) atomicMax(longest, best);
}

// parts[g * (kMaxParts + 1) + i]: columns that cut granule g into kMaxParts ranges with about equally many entries of the
// longest row of B (of equal width where that row has few).
__global__ void k_granule_parts(const int32_t* __restrict__ b_col, const u32* __restrict__ bound, const u64* __restrict__ longest,
                                int granules, int log2_g, u32* __restrict__ parts) {
  const int g = blockIdx.x, i = threadIdx.x;
  if (i > kMaxParts) return;
  const u32 k = static_cast<u32>(*longest);
  const u32 s = bound[static_cast<i64>(k) * (granules + 1) + g], e = bound[static_cast<i64>(k) * (granules + 1) + g + 1];
  const u32 lo = static_cast<u32>(g) << log2_g, w = 1u << log2_g;
  u32 c = lo + static_cast<u32>((static_cast<u64>(w) * i) / kMaxParts);
  if (e - s >= 8 * kMaxParts && i > 0 && i < kMaxParts) c = static_cast<u32>(b_col[s + static_cast<u32>((static_cast<u64>(e - s) * i) / kMaxParts)]);
  parts[g * (kMaxParts + 1) + i] = c;
}

// Products of every heavy row per granule.  A warp per row; rows with more than kCountLong entries are listed and taken by
// k_granule_counts_long, many blocks per row.
constexpr u32 kCountLong = 1024;
__device__ __forceinline__ void count_granules(const int32_t* __restrict__ a_col, i64 s, i64 e, const u32* __restrict__ bound, int granules,
                                               u32* __restrict__ out, bool add) {
  const int lane = threadIdx.x & 31;
  const int width = granules >= 32 ? 32 : granules;  // (a power of two)
  const int sub = lane / width, step = 32 / width;
  for (int c0 = 0; c0 < granules; c0 += 32) {
    const int c = c0 + (lane & (width - 1));
    u32 sum = 0;
    if (add) {  // (a slice of a long row: many warps, one after the other)
#pragma unroll 4
      for (i64 j = s + sub; j < e; j += step) {
        const u32* bp = bound + static_cast<i64>(a_col[j]) * (granules + 1) + c;
        sum += bp[1] - bp[0];
      }
    }
    for (i64 j0 = s; !add && j0 < e; j0 += 32) {  // 32 entries' columns at once, so that the look-ups do not wait for one another
      const int n = static_cast<int>(min(i64{32}, e - j0));
      const int32_t mine = lane < n ? a_col[j0 + lane] : 0;
#pragma unroll 8
      for (int t = 0; t < n; t += step) {
        const int32_t k = __shfl_sync(0xffffffffu, mine, t + sub);
        if (t + sub < n) {
          const u32* bp = bound + static_cast<i64>(k) * (granules + 1) + c;
          sum += bp[1] - bp[0];
        }
      }
    }
    for (int o = width; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (sub == 0) {
      if (!add) out[c] = sum;
      else if (sum) atomicAdd(&out[c], sum);
    }
  }
}
__global__ void __launch_bounds__(256) k_granule_counts(const int32_t* __restrict__ x_heavy, i64 n_heavy, const i64* __restrict__ a_row_ptr,
                                                        const int32_t* __restrict__ a_col, const u32* __restrict__ bound, int granules,
                                                        u32* __restrict__ counts, int32_t* __restrict__ long_rows, u32* __restrict__ n_long,
                                                        const unsigned char* __restrict__ in_panel) {
  const i64 n_warps = static_cast<i64>(gridDim.x) * 8;
  for (i64 h = static_cast<i64>(blockIdx.x) * 8 + (threadIdx.x >> 5); h < n_heavy; h += n_warps) {
    if (in_panel && in_panel[h]) continue;
    const i64 row = x_heavy[h];
    const i64 s = a_row_ptr[row], e = a_row_ptr[row + 1];
    if (e - s > kCountLong) {
      for (int c = threadIdx.x & 31; c < granules; c += 32) counts[h * granules + c] = 0;
      if ((threadIdx.x & 31) == 0) long_rows[atomicAdd(n_long, 1u)] = static_cast<int32_t>(h);
    } else {
      count_granules(a_col, s, e, bound, granules, counts + h * granules, false);
    }
  }
}
// The blocks form groups, one row at a time to a group, and the blocks of a group take the row's runs of kCountRun entries in turn, a
// slice per warp: kCountRuns blocks to a group, or as many more as few rows leave.  (With all warps of the grid round-robin over all
// slices, every warp looked up every row's ends, one after the other: 730 us of R-MAT scale 19.  With kCountRuns blocks however few the
// rows: one row of 10^6 entries 750 us, two of 300000 255, now 34 and 35.)
constexpr int kCountRun = 8 * 256, kCountRuns = 16;
__global__ void __launch_bounds__(256) k_granule_counts_long(const int32_t* __restrict__ x_heavy, const i64* __restrict__ a_row_ptr,
                                                             const int32_t* __restrict__ a_col, const u32* __restrict__ bound, int granules,
                                                             u32* __restrict__ counts, const int32_t* __restrict__ long_rows,
                                                             const u32* __restrict__ n_long) {
  const u32 n = *n_long;
  if (n == 0) return;
  const u32 groups = min(n, gridDim.x / kCountRuns), blocks = gridDim.x / groups, run = blockIdx.x % blocks;
  if (blockIdx.x / blocks >= groups) return;  // (left over)
  for (u32 q = blockIdx.x / blocks; q < n; q += groups) {
    const i64 h = long_rows[q];
    const i64 row = x_heavy[h];
    const i64 e = a_row_ptr[row + 1];
    for (i64 s = a_row_ptr[row] + static_cast<i64>(run) * kCountRun + (threadIdx.x >> 5) * 256; s < e; s += static_cast<i64>(blocks) * kCountRun)
      count_granules(a_col, s, min(e, s + 256), bound, granules, counts + h * granules, true);
  }
}

// Walks a row's granules from left to right and calls emit(first granule, granules, products, parts) per range; returns
// the number of tasks.
template <typename Emit>
__device__ __forceinline__ u32 cut_row(const u32* __restrict__ counts, u32 products, const TaskRules& r, Emit emit) {
  u32 tasks = 0;
  int g = 0;
  u32 left = products;
  while (left > 0) {
    u32 n = r.granules == 1 ? products : counts[g];
    if (n == 0) { ++g; continue; }
    int w = 1;
    // one more granule while a warp, or a mid-size block, can still take the whole
    while (g + w < r.granules && n < left) {
      const u32 more = counts[g + w];
      const u32 sum = n + more, width = static_cast<u32>(w + 1) << r.log2_g;
      const bool fits = (sum <= static_cast<u32>(r.small_max) && width <= r.small_width) ||
                        (sum <= static_cast<u32>(r.mid_max) && width <= r.mid_width);
      if (!fits) break;
      n = sum;
      ++w;
    }
    u32 parts = 1;
    if (w == 1 && n > r.split_above)
      while (parts < static_cast<u32>(r.max_parts) && n / parts > r.split_above) parts *= 2;
    emit(g, w, n, parts);
    tasks += parts;
    left -= n;
    g += w;
  }
  return tasks;
}

__global__ void __launch_bounds__(128) k_task_count(const u32* __restrict__ counts, const i64* __restrict__ heavy_base, i64 n_heavy,
                                                    TaskRules r, u32* __restrict__ row_tasks, const unsigned char* __restrict__ in_panel,
                                                    const u64* __restrict__ panels, u64* __restrict__ host_panels) {
  const i64 h = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (panels && h < kPanelCounts) host_panels[h] = panels[h];  // (read after a synchronisation)
  if (h >= n_heavy) return;
  if (in_panel && in_panel[h]) row_tasks[h] = 1;
  else row_tasks[h] = cut_row(counts + h * r.granules, static_cast<u32>(heavy_base[h + 1] - heavy_base[h]), r, [](int, int, u32, u32) {});
}

// Where the tasks of a batch go.  lists: [0] small, [1] mid, [2] big (the huge ones from the front of the batch's part of the
// list, the others from its back); counters: [0] small, [1] mid, [2] huge, [3] other big.
struct TaskTables {
  HeavyTask* tasks;
  i64* task_off;
  int32_t* list[3];
  int* counters;
  i64 first, end;  // the batch's part of the tables
};

// Class of a range (an index into TaskTables::counters).
__device__ __forceinline__ int class_of(const TaskRules& r, int granules, u32 n, u32 parts) {
  if (parts > 1) return 2;
  if (n <= static_cast<u32>(r.small_max)) return 0;
  if (n <= static_cast<u32>(r.mid_max) && static_cast<u32>(granules) << r.log2_g <= r.mid_width) return 1;
  return n > static_cast<u32>(kHugeChunk) ? 2 : 3;
}

// Writes the tasks of heavy row h, the first of them at position id.  place(c): next position of class c.
template <typename Place>
__device__ __forceinline__ void emit_row(const u32* __restrict__ counts, const i64* __restrict__ heavy_base, i64 h, i64 elem0,
                                         const TaskRules& r, i64 id, const int32_t* __restrict__ x_heavy,
                                         const i64* __restrict__ a_row_ptr, const u32* __restrict__ parts_tab, const TaskTables& tt,
                                         const unsigned char* __restrict__ in_panel, Place place) {
  const i64 row = x_heavy[h];
  HeavyTask t;
  t.a0 = a_row_ptr[row];
  t.n_a = static_cast<u32>(a_row_ptr[row + 1] - t.a0);
  i64 off = heavy_base[h] - elem0;
  auto put = [&](int cls) {
    const int b = static_cast<int>(id - tt.first);  // lists hold batch-relative ids
    if (cls == 0 || cls == 1) tt.list[cls][tt.first + place(cls)] = b;
    else if (cls == 2) tt.list[2][tt.first + place(2)] = b;
    else if (cls == 3) tt.list[2][tt.end - 1 - place(3)] = b;
    tt.tasks[id] = t;
    tt.task_off[id] = t.off;
    ++id;
  };
  if (in_panel && in_panel[h]) {
    t.lo = 0;
    t.hi = static_cast<u32>(r.granules) << r.log2_g;
    t.off = off;
    t.n = static_cast<u32>(heavy_base[h + 1] - heavy_base[h]);
    put(-1);  // (a panel's row is in no list)
    return;
  }
  cut_row(counts + h * r.granules, static_cast<u32>(heavy_base[h + 1] - heavy_base[h]), r, [&](int g, int w, u32 n, u32 parts) {
    const u32 lo = static_cast<u32>(g) << r.log2_g;
    const u32 width = static_cast<u32>(w) << r.log2_g;
    if (parts > 1) {
      const u32* cut = parts_tab + g * (kMaxParts + 1);
      for (u32 i = 0; i < parts; ++i) {
        t.lo = cut[i * (kMaxParts / parts)];
        t.hi = cut[(i + 1) * (kMaxParts / parts)];
        t.off = off + (t.lo - lo);
        t.n = 0;
        put(2);
      }
    } else {
      t.lo = lo;
      t.hi = lo + width;
      t.off = off;
      t.n = n;
      put(class_of(r, w, n, 1));
    }
    off += n;
  });
}

// Rows h0 .. h1 - 1 (a batch).  row_task_off: exclusive prefix sums of row_tasks.
__global__ void __launch_bounds__(128) k_task_emit(const u32* __restrict__ counts, const i64* __restrict__ heavy_base, i64 h0, i64 h1,
                                                   i64 elem0, TaskRules r, const i64* __restrict__ row_task_off,
                                                   const int32_t* __restrict__ x_heavy, const i64* __restrict__ a_row_ptr,
                                                   const u32* __restrict__ parts_tab, TaskTables tt,
                                                   const unsigned char* __restrict__ in_panel) {
  // Places in the lists are drawn once per block and class.  With an atomic per task on four words of L2, which take turns, this kernel
  // took 112 us for R-MAT scale 17 (now 27) and 1.5 ms for scale 19.
  __shared__ u32 s_n[4], s_base[4];
  const i64 h = h0 + static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool mine = h < h1;
  if (threadIdx.x < 4) s_n[threadIdx.x] = 0u;
  __syncthreads();
  if (mine && !(in_panel && in_panel[h])) {
    u32 n_of[4] = {0u, 0u, 0u, 0u};
    cut_row(counts + h * r.granules, static_cast<u32>(heavy_base[h + 1] - heavy_base[h]), r, [&](int, int w, u32 n, u32 parts) {
      const int c = class_of(r, w, n, parts);
#pragma unroll
      for (int i = 0; i < 4; ++i) n_of[i] += i == c ? parts : 0u;
    });
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (n_of[i]) atomicAdd(&s_n[i], n_of[i]);
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    s_base[threadIdx.x] = s_n[threadIdx.x] ? static_cast<u32>(atomicAdd(&tt.counters[threadIdx.x], static_cast<int>(s_n[threadIdx.x]))) : 0u;
    s_n[threadIdx.x] = 0u;
  }
  __syncthreads();
  if (mine)
    emit_row(counts, heavy_base, h, elem0, r, row_task_off[h], x_heavy, a_row_ptr, parts_tab, tt, in_panel,
             [&](int c) { return s_base[c] + atomicAdd(&s_n[c], 1u); });
}

// ---------------------------------------------------------------------------------------------------------------------
// what the kernels share
// ---------------------------------------------------------------------------------------------------------------------
template <typename V>
struct TaskInput {
  const int32_t* a_col;
  const V* a_val;
  const int32_t* b_col;
  const V* b_val;
  const u32* bound;
  int granules, log2_g;
};

// The piece of row k of B inside the task's columns: positions [start, end).
template <typename V>
__device__ __forceinline__ void find_piece(const TaskInput<V>& in, int32_t k, u32 lo, u32 hi, u32& start, u32& end) {
  const u32 g = 1u << in.log2_g;
  const u32* bp = in.bound + static_cast<i64>(k) * (in.granules + 1);
  const u32 c0 = lo >> in.log2_g, c1 = (hi + g - 1) >> in.log2_g;
  start = bp[c0];
  end = bp[c1];
  if (((lo | hi) & (g - 1)) != 0) {  // (uniform: a sub-range of one granule)
    u32 a = start, b = end;
    while (a < b) {
      const u32 m = a + ((b - a) >> 1);
      if (static_cast<u32>(in.b_col[m]) >= lo) b = m; else a = m + 1;
    }
    start = a;
    b = end;
    while (a < b) {
      const u32 m = a + ((b - a) >> 1);
      if (static_cast<u32>(in.b_col[m]) >= hi) b = m; else a = m + 1;
    }
    end = a;
  }
}

// Debug mode: every product of heavy row h (a block each) lies in the columns of exactly one task.  The tasks' ranges ascend
// and do not overlap, the entries of every piece lie in its task's columns, and the pieces hold the row's products.
template <typename V>
__global__ void __launch_bounds__(256) k_validate_tasks(TaskInput<V> in, const HeavyTask* __restrict__ tasks, const i64* __restrict__ row_task_off,
                                                        const i64* __restrict__ heavy_base, i64 n_heavy, i64 n_cols, int* __restrict__ err) {
  __shared__ i64 s_sum[33];
  for (i64 h = blockIdx.x; h < n_heavy; h += gridDim.x) {
    i64 sum = 0;
    bool bad = false;
    u32 from = 0;
    for (i64 id = row_task_off[h]; id < row_task_off[h + 1]; ++id) {
      const HeavyTask t = tasks[id];
      bad |= t.lo < from || t.hi <= t.lo;
      from = t.hi;
      const i64 before = sum;
      for (u32 j = threadIdx.x; j < t.n_a; j += 256) {
        u32 a, b;
        find_piece(in, in.a_col[t.a0 + j], t.lo, t.hi, a, b);
        for (u32 q = a; q < b; ++q) {
          const i64 c = in.b_col[q];
          bad |= c < static_cast<i64>(t.lo) || c >= static_cast<i64>(t.hi) || c >= n_cols;
        }
        sum += static_cast<i64>(b) - static_cast<i64>(a);
      }
      i64 n;
      block_exclusive_scan(sum - before, s_sum, &n);
      __syncthreads();
      bad |= t.n != 0 && n != static_cast<i64>(t.n);  // (0: a sub-range, not counted)
    }
    i64 n;
    block_exclusive_scan(sum, s_sum, &n);
    __syncthreads();
    if (bad || n != heavy_base[h + 1] - heavy_base[h]) dev_set_error(err, kDevBadChunk);
  }
}

// The non-empty pieces of a round of rows of B, in shared memory: piece q holds the products [ex[q], ex[q + 1]) of the
// round, and product f of it is the entry at position base[q] + f of B, times a[q].
template <typename V, int CAP>
struct Pieces {
  V a[CAP];
  u32 base[CAP];
  int ex[CAP + 33];  // (the lanes of a warp look up to 32 pieces ahead)
};
struct RoundSize {
  int pieces, products;
};

// The products of a round that fall to warp `warp` of `n_warps`: a contiguous, equal share, 32 at a time and U times that in
// flight: load(u, position in B, a) for the valid lanes of U windows, then use(u, valid, number of the product in the round) for each.  `load` only requests;
// arithmetic on what it loads would wait there, window after window.
// Every lane finds its piece from the ones that start inside the windows, all U windows at once: the chain from one round of U
// windows to the next is one look at the piece starts and a population count.  (Window after window, with a way of its own for
// windows inside one piece, the chain of four dependent shared-memory loads per window bound the mid-size tasks: R-MAT scale 19
// fp32 27.0 ms against 23.1, scale 17 fp64 1.66 against 1.52, block-dense fp32 0.65 against 0.51.  A second set of windows
// requested before the first is used: 27.9, the registers cost more.  Windows that end with their piece, the remaining
// lanes idle: 37.7.)
template <typename V, int CAP, int U, typename Load, typename Use>
__device__ __forceinline__ void walk_products(const Pieces<V, CAP>& pc, const RoundSize& rs, int warp, int n_warps, Load load, Use use) {
  int f = static_cast<int>((static_cast<i64>(rs.products) * warp) / n_warps);
  const int f1 = static_cast<int>((static_cast<i64>(rs.products) * (warp + 1)) / n_warps);
  if (f >= f1) return;
  const int lane = threadIdx.x & 31;
  const u32 upto = lanemask_lt() | (1u << lane);
  int cur = 0;
  for (int hi = rs.pieces - 1; cur < hi;) {  // last piece that starts at or before f
    const int mid = (cur + hi + 1) >> 1;
    if (pc.ex[mid] <= f) cur = mid; else hi = mid - 1;
  }
  for (; f < f1; f += U * 32) {
    // pieces that start inside the U windows, as masks over the windows' positions
    u32 heads[U];
#pragma unroll
    for (int u = 0; u < U; ++u) heads[u] = 0u;
    for (int i = cur + 1 + lane;; i += 32) {
      const u32 d = static_cast<u32>(pc.ex[i] - f);
      if (U <= 2 && !__any_sync(0xffffffffu, d < U * 32u)) break;  // (inside one piece; four windows seldom are)
#pragma unroll
      for (int u = 0; u < U; ++u) heads[u] |= __reduce_or_sync(0xffffffffu, d - u * 32 < 32u ? 1u << (d & 31) : 0u);
      if (!__all_sync(0xffffffffu, d < U * 32u)) break;  // (usually at once; ex is sorted)
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = cur + __popc(heads[u] & upto);
      const int g = f + u * 32 + lane;
      if (g < f1) load(u, pc.base[q] + static_cast<u32>(g), pc.a[q]);
      cur += __popc(heads[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (f + u * 32 < f1) use(u, f + u * 32 + lane < f1, f + u * 32 + lane);
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// small tasks: one warp each
// ---------------------------------------------------------------------------------------------------------------------
template <typename V, int K, int KMAX>
__device__ __forceinline__ int small_task(const TaskInput<V>& in, const HeavyTask& t, int32_t* __restrict__ out_col, V* __restrict__ out_val,
                                          u32* s_base, V* s_a, u32* s_key, V* s_val) {
  constexpr int kPosBits = 5 + (K == 1 ? 0 : K == 2 ? 1 : K == 4 ? 2 : K == 8 ? 3 : 4);
  constexpr int U = K >= 4 ? 4 : K;
  const int lane = threadIdx.x & 31;
  int done = 0;
  for (u32 j0 = 0; j0 < t.n_a; j0 += 32) {
    const u32 j = j0 + lane;
    u32 start = 0, end = 0;
    V av = V(0);
    if (j < t.n_a) {
      const int32_t k = in.a_col[t.a0 + j];
      av = in.a_val[t.a0 + j];
      find_piece(in, k, t.lo, t.hi, start, end);
    }
    const int len = static_cast<int>(end - start);
    const u32 some = __ballot_sync(0xffffffffu, len > 0);
    if (!some) continue;
    const int inc = warp_inclusive_scan(len);
    const int ex = inc - len;
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    if (len > 0) {
      const int p = __popc(some & lanemask_lt());
      s_base[p] = start - static_cast<u32>(ex);
      s_a[p] = av;
    }
    __syncwarp();
    int started = 0;
    for (int f0 = 0; f0 < total; f0 += 32 * U) {
      u32 c[U];
      V v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int w = ex - (f0 + u * 32);
        const u32 heads = __reduce_or_sync(0xffffffffu, (len > 0 && w >= 0 && w < 32) ? 1u << w : 0u);
        const int f = f0 + u * 32 + lane;
        if (f < total) {
          const int q = started + __popc(heads & (lanemask_lt() | (1u << lane))) - 1;
          const u32 src = s_base[q] + static_cast<u32>(f);
          c[u] = static_cast<u32>(in.b_col[src]) - t.lo;
          v[u] = in.b_val[src] * s_a[q];
        }
        started += __popc(heads);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int f = f0 + u * 32 + lane;
        if (f < total) {
          s_key[done + f] = (c[u] << kPosBits) | static_cast<u32>(done + f);
          s_val[done + f] = v[u];
        }
      }
    }
    done += total;
    __syncwarp();
  }
  u32 key[K];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int q = r * 32 + lane;
    key[r] = q < done ? s_key[q] : 0xffffffffu;
  }
  __syncwarp();
  warp_sort_keys<u32, K>(key, lane);
  const int m = warp_sum_runs<V, u32, K, kPosBits>(key, done, s_key, s_val, t.lo, out_col + t.off, out_val + t.off);
  __syncwarp();
  return m;
}

template <typename V, int KMAX>
__global__ void __launch_bounds__(kSmallWarps * 32, KMAX > 4 ? 8 : 10) k6_small_tasks(
    TaskInput<V> in, const HeavyTask* __restrict__ tasks, const int32_t* __restrict__ list, const int* __restrict__ counters,
    int32_t* __restrict__ out_col, V* __restrict__ out_val, u32* __restrict__ task_nnz,
    u64* __restrict__ totals) {  // [0] += products, [1] += entries (statistics)
  __shared__ u32 s_base[kSmallWarps][32];
  __shared__ V s_a[kSmallWarps][32];
  __shared__ __align__(16) u32 s_key[kSmallWarps][32 * KMAX];
  __shared__ V s_val[kSmallWarps][32 * KMAX];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_list = counters[0];
  const int step = gridDim.x * kSmallWarps;
  u64 sum_n = 0, sum_m = 0;
  for (int q = blockIdx.x * kSmallWarps + w; q < n_list; q += step) {
    const int id = list[q];
    const HeavyTask t = tasks[id];
    int m;
    if (t.n <= 32) m = small_task<V, 1, KMAX>(in, t, out_col, out_val, s_base[w], s_a[w], s_key[w], s_val[w]);
    else if (t.n <= 64) m = small_task<V, 2, KMAX>(in, t, out_col, out_val, s_base[w], s_a[w], s_key[w], s_val[w]);
    else if (KMAX == 4 || t.n <= 128) m = small_task<V, 4, KMAX>(in, t, out_col, out_val, s_base[w], s_a[w], s_key[w], s_val[w]);
    else if (t.n <= 256) m = small_task<V, (KMAX > 4 ? 8 : 4), KMAX>(in, t, out_col, out_val, s_base[w], s_a[w], s_key[w], s_val[w]);
    else m = small_task<V, (KMAX > 4 ? 16 : 4), KMAX>(in, t, out_col, out_val, s_base[w], s_a[w], s_key[w], s_val[w]);
    if (lane == 0) {
      task_nnz[id] = static_cast<u32>(m);
      sum_n += t.n;
      sum_m += static_cast<u32>(m);
    }
  }
  if (lane == 0 && sum_n) {
    atomicAdd(&totals[0], sum_n);
    atomicAdd(&totals[1], sum_m);
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// mid and big tasks: rounds of rows of B, shared by a block
// ---------------------------------------------------------------------------------------------------------------------
// A round's rows of B in registers: PER per thread.
template <typename V, int PER>
struct PieceRegs {
  u32 start[PER], end[PER];
  int32_t k[PER];
  V a[PER];
};
template <typename V, int T, int PER>
__device__ __forceinline__ void load_rows(const TaskInput<V>& in, const HeavyTask& t, u32 round, PieceRegs<V, PER>& r) {
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const u32 j = (round * PER + i) * T + threadIdx.x;
    r.k[i] = -1;
    if (j < t.n_a) {
      r.k[i] = in.a_col[t.a0 + j];
      r.a[i] = in.a_val[t.a0 + j];
    }
  }
}
template <typename V, int PER>
__device__ __forceinline__ void load_pieces(const TaskInput<V>& in, const HeavyTask& t, PieceRegs<V, PER>& r) {
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    r.start[i] = r.end[i] = 0;
    if (r.k[i] >= 0) find_piece(in, r.k[i], t.lo, t.hi, r.start[i], r.end[i]);
  }
}
// Registers -> shared memory.  The caller's barrier before it: the pieces of the round before are no longer read.  Ends
// with a barrier.
template <typename V, int T, int PER>
__device__ __forceinline__ RoundSize build_pieces(const PieceRegs<V, PER>& r, Pieces<V, T * PER>& pc, uint2* s_sum) {
  constexpr int kWarps = T / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  u32 n_mine = 0, p_mine = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const u32 len = r.end[i] - r.start[i];
    n_mine += len;
    p_mine += len ? 1u : 0u;
  }
  u32 n_inc = 0, p_inc = 0;
  if (__any_sync(0xffffffffu, n_mine != 0)) {  // (most rows of A fill a few warps)
    n_inc = warp_inclusive_scan(n_mine);
    p_inc = warp_inclusive_scan(p_mine);
  }
  if (lane == 31) s_sum[warp] = make_uint2(n_inc, p_inc);
  __syncthreads();
  const uint2 w = lane < kWarps ? s_sum[lane] : make_uint2(0, 0);
  RoundSize rs;
  rs.products = static_cast<int>(__reduce_add_sync(0xffffffffu, w.x));
  rs.pieces = static_cast<int>(__reduce_add_sync(0xffffffffu, w.y));
  if (__any_sync(0xffffffffu, n_mine != 0)) {
    u32 ex = __reduce_add_sync(0xffffffffu, lane < warp ? w.x : 0u) + n_inc - n_mine;
    u32 q = __reduce_add_sync(0xffffffffu, lane < warp ? w.y : 0u) + p_inc - p_mine;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const u32 len = r.end[i] - r.start[i];
      if (len) {
        pc.ex[q] = static_cast<int>(ex);
        pc.base[q] = r.start[i] - ex;
        pc.a[q] = r.a[i];
        ++q;
        ex += len;
      }
    }
  }
  if (tid < 33) pc.ex[rs.pieces + tid] = tid == 0 ? rs.products : INT_MAX;
  __syncthreads();
  return rs;
}

// Tasks are handed out by a ticket over a list; thread 0 keeps the chain ticket -> list entry -> task record of the next
// ones in flight (see TaskPipe).
struct TaskFeed {
  int* ticket;
  int n_list, n_front;
  const int32_t* list;
  i64 list_flip;  // >= 0: list positions past n_front are read from the back
  const HeavyTask* tasks;
  int tk2 = 0, tk3 = 0;
  int k1 = -1, k2 = -1;
  HeavyTask next;

  __device__ __forceinline__ int list_at(int t) const {
    if (t >= n_list) return -1;
    return (list_flip < 0 || t < n_front) ? list[t] : list[list_flip - (t - n_front)];
  }
  __device__ __forceinline__ void start(int* id, HeavyTask* first) {
    const int t0 = atomicAdd(ticket, 3);
    const int k0 = list_at(t0);
    k1 = list_at(t0 + 1);
    tk2 = t0 + 2;
    *id = k0;
    if (k0 >= 0) *first = tasks[k0];
  }
  __device__ __forceinline__ void issue() {  // start of a task
    tk3 = atomicAdd(ticket, 1);
    k2 = list_at(tk2);
    if (k1 >= 0) next = tasks[k1];
  }
  __device__ __forceinline__ void publish(int* id, HeavyTask* t) {  // when the task's products are done
    *id = k1;
    *t = next;
    k1 = k2;
    tk2 = tk3;
  }
};

// ---------------------------------------------------------------------------------------------------------------------
// mid tasks: symbolic pass, ranks, numeric pass
// ---------------------------------------------------------------------------------------------------------------------
// Per block: bitmap of the task's columns | rank of every word's first entry | compact values | compact columns.  Pass 1
// marks the columns (and keeps the products, if they fit the half of the arrays that the entries do not take), a prefix sum over the
// words ranks them, pass 2 adds every product to the slot of its column's rank and notes the column; the write-out is one coalesced
// copy.
constexpr int kMidPerThread = 2;    // rows of B per thread and round
// Windows of 32 products a warp has in flight (fp64: with four the registers spill, 1.35 against 1.19 ms for the big tasks
// of R-MAT scale 17, 1.89 against 1.67 for the mid ones).
template <typename V> constexpr int kMidUnroll = 16 / sizeof(V);

inline size_t mid_task_smem_bytes(int width, int val_bytes, int entries) {
  const size_t n_words = static_cast<size_t>(width) / 32;
  return ((n_words * 6 + 15) & ~size_t{15}) + static_cast<size_t>(entries) * (val_bytes + 2) + 64;
}

template <typename V>
__global__ void __launch_bounds__(kMidThreads, 6) k6_mid_tasks(
    TaskInput<V> in, const HeavyTask* __restrict__ tasks, const int32_t* __restrict__ list, const int* __restrict__ n_list, int* ticket,
    int width, int entries, int32_t* __restrict__ out_col, V* __restrict__ out_val, u32* __restrict__ task_nnz,
    u64* __restrict__ totals) {  // [0] += products, [1] += entries (statistics)
  extern __shared__ __align__(16) unsigned char smem_mid_raw[];
  constexpr int T = kMidThreads, PER = kMidPerThread, U = kMidUnroll<V>;
  constexpr int kWarps = T / 32;
  constexpr int CAP = T * PER;
  const int n_words = width >> 5;
  u32* bitmap = reinterpret_cast<u32*>(smem_mid_raw);                          // n_words
  unsigned short* wpre = reinterpret_cast<unsigned short*>(bitmap + n_words);  // n_words: rank of the word's first entry
  V* oval = reinterpret_cast<V*>(smem_mid_raw + ((static_cast<size_t>(n_words) * 6 + 15) & ~size_t{15}));
  unsigned short* ocol = reinterpret_cast<unsigned short*>(oval + entries);    // the entries' columns relative to the task's first
  __shared__ Pieces<V, CAP> pc;
  __shared__ uint2 s_sum[kWarps];
  __shared__ u32 s_wsum[kWarps];
  __shared__ HeavyTask s_task[2];
  __shared__ int s_id[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wpt = n_words > T ? n_words / T : 1;
  const int wb = tid * wpt;
  const bool own = wb < n_words;

  for (int w = tid; w < n_words; w += T) bitmap[w] = 0u;
  for (int i = tid; i < entries; i += T) oval[i] = V(0);
  TaskFeed feed{ticket, *n_list, 0, list, -1, tasks};
  if (tid == 0) feed.start(&s_id[0], &s_task[0]);
  __syncthreads();
  u64 sum_n = 0, sum_m = 0;
  int par = 0;
  int id = s_id[0];
  HeavyTask task = s_task[0];
  PieceRegs<V, PER> regs;
  if (id >= 0) {
    load_rows<V, T, PER>(in, task, 0, regs);
    load_pieces<V, PER>(in, task, regs);
  }

  while (id >= 0) {
    const int n_rounds = static_cast<int>((task.n_a + CAP - 1) / CAP);
    if (tid == 0) feed.issue();
    const u32 lo = task.lo;
    u32 c[U];
    V v[U], av[U];
    RoundSize rs = build_pieces<V, T, PER>(regs, pc, s_sum);
    // Products that fill at most half of the compact arrays wait in the other half for pass 2, which then neither walks the pieces nor
    // loads anything: this kernel 5.82 -> 5.47 ms for R-MAT scale 18 fp32, the call 59.1 -> 57.4 for scale 19.  (Larger arrays, for all of
    // the class, leave four blocks an SM: 63.8; tasks cut so that more of them fit: 57.7.)
    const int half = entries / 2;
    const bool keep = task.n <= static_cast<u32>(half);
    V* const kept_val = oval + half;
    unsigned short* const kept_col = ocol + half;
    int before = 0;  // products of the rounds before

    // ---- pass 1 (symbolic): mark the columns
    auto mark = [&](u32 c) {
      const u32 bit = 1u << (c & 31);
      u32* const w = &bitmap[c >> 5];
      if (!(*w & bit)) atomicOr(w, bit);  // (lanes with neighbouring columns share a word, and atomics on it take turns)
    };
    for (int r = 0;;) {
      const bool more = ++r < n_rounds;
      if (more) load_rows<V, T, PER>(in, task, r, regs);
      if (keep)
        walk_products<V, CAP, U>(
            pc, rs, warp, kWarps,
            [&](int u, u32 src, V a) {
              c[u] = static_cast<u32>(in.b_col[src]);
              v[u] = in.b_val[src];
              av[u] = a;
            },
            [&](int u, bool valid, int f) {
              if (valid) {
                mark(c[u] - lo);
                kept_col[before + f] = static_cast<unsigned short>(c[u] - lo);
                kept_val[before + f] = av[u] * v[u];
              }
            });
      else
        walk_products<V, CAP, U>(
            pc, rs, warp, kWarps, [&](int u, u32 src, V) { c[u] = static_cast<u32>(in.b_col[src]); },
            [&](int u, bool valid, int) { if (valid) mark(c[u] - lo); });
      before += rs.products;
      if (!more) break;
      load_pieces<V, PER>(in, task, regs);
      __syncthreads();
      rs = build_pieces<V, T, PER>(regs, pc, s_sum);
    }
    __syncthreads();
    // ---- ranks: exclusive prefix over the words' populations
    u32 pop = 0;
    uint4 b0 = make_uint4(0, 0, 0, 0), b1 = b0;  // the usual case: eight words per thread
    if (own) {
      if (wpt == 8) {
        b0 = *reinterpret_cast<const uint4*>(bitmap + wb);
        b1 = *reinterpret_cast<const uint4*>(bitmap + wb + 4);
        pop = __popc(b0.x) + __popc(b0.y) + __popc(b0.z) + __popc(b0.w) + __popc(b1.x) + __popc(b1.y) + __popc(b1.z) + __popc(b1.w);
      } else {
        for (int i = 0; i < wpt; ++i) pop += __popc(bitmap[wb + i]);
      }
    }
    const u32 inc = warp_inclusive_scan(pop);
    if (lane == 31) s_wsum[warp] = inc;
    __syncthreads();
    u32 ex = inc - pop, total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const u32 ws = s_wsum[w];
      if (w < warp) ex += ws;
      total += ws;
    }
    if (own) {
      if (wpt == 8) {
        u32 r0 = ex, r1 = r0 + __popc(b0.x), r2 = r1 + __popc(b0.y), r3 = r2 + __popc(b0.z), r4 = r3 + __popc(b0.w);
        u32 r5 = r4 + __popc(b1.x), r6 = r5 + __popc(b1.y), r7 = r6 + __popc(b1.z);
        *reinterpret_cast<uint4*>(wpre + wb) = make_uint4(r0 | (r1 << 16), r2 | (r3 << 16), r4 | (r5 << 16), r6 | (r7 << 16));
      } else {
        u32 run = ex;
        for (int i = 0; i < wpt; ++i) {
          wpre[wb + i] = static_cast<unsigned short>(run);
          run += __popc(bitmap[wb + i]);
        }
      }
    }
    if (tid == 0) feed.publish(&s_id[par ^ 1], &s_task[par ^ 1]);
    __syncthreads();
    const int next_id = s_id[par ^ 1];
    const HeavyTask next = s_task[par ^ 1];
    // ---- pass 2 (numeric): every product to the slot of its column's rank
    auto put = [&](u32 c, V v) {
      const u32 r = static_cast<u32>(wpre[c >> 5]) + __popc(bitmap[c >> 5] & ((1u << (c & 31)) - 1u));
      atomicAdd(&oval[r], v);
      ocol[r] = static_cast<unsigned short>(c);  // (every product of the column writes the same value)
    };
    if (keep) {
      for (int i = tid; i < static_cast<int>(task.n); i += T) {
        put(kept_col[i], kept_val[i]);
        kept_val[i] = V(0);  // (the slots of a larger task)
      }
    }
    for (int r = 0; !keep && r < n_rounds; ++r) {
      if (n_rounds > 1) {
        if (r > 0) __syncthreads();  // (the first time the pieces of the last round are no longer read either)
        load_rows<V, T, PER>(in, task, r, regs);
        load_pieces<V, PER>(in, task, regs);
        rs = build_pieces<V, T, PER>(regs, pc, s_sum);
      }
      walk_products<V, CAP, U>(
          pc, rs, warp, kWarps,
          [&](int u, u32 src, V a) {
            c[u] = static_cast<u32>(in.b_col[src]);
            v[u] = in.b_val[src];
            av[u] = a;
          },
          [&](int u, bool valid, int) { if (valid) put(c[u] - lo, av[u] * v[u]); });
    }
    // the next task's first rows of B are requested before this task is written out
    if (next_id >= 0) load_rows<V, T, PER>(in, next, 0, regs);
    __syncthreads();
    if (next_id >= 0) load_pieces<V, PER>(in, next, regs);
    if ((n_words & 3) == 0) {
      for (int w = tid * 4; w < n_words; w += T * 4) *reinterpret_cast<uint4*>(bitmap + w) = make_uint4(0, 0, 0, 0);
    } else {
      for (int w = tid; w < n_words; w += T) bitmap[w] = 0u;
    }
    int32_t* const col = out_col + task.off;
    V* const val = out_val + task.off;
    for (int i = tid; i < static_cast<int>(total); i += T) {
      col[i] = static_cast<int32_t>(lo + ocol[i]);
      val[i] = oval[i];
      oval[i] = V(0);
    }
    if (tid == 0) {
      task_nnz[id] = total;
      sum_n += task.n;
      sum_m += total;
    }
    __syncthreads();
    task = next;
    id = next_id;
    par ^= 1;
  }
  if (tid == 0 && sum_n) {
    atomicAdd(&totals[0], sum_n);
    atomicAdd(&totals[1], sum_m);
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// big tasks: the dense accumulator
// ---------------------------------------------------------------------------------------------------------------------
// One value per column of the granule.  An idle slot holds -0.0, the identity of the addition, and a product that is a zero
// of either sign is added as +0.0, so that a slot that received anything is never -0.0 again: which columns have an entry
// is read off the values, and a product costs one shared-memory add and nothing else.  (Rounded to the product first, then
// +0.0 added: fma(a, b, +0.0) is -0.0 where a negative product underflows, and the column would have no entry.)  The flush goes over the granule twice: every warp
// counts the entries of its share, the block adds the counts up, and the warp writes its share, a 16-byte word per lane at a
// time (128 columns in fp32; 32 columns at a time took 36 instructions for each 32).
// Bank spreading: the low bits of a power-law matrix's columns are mostly zero; the slot of a column inside its group of
// 32 is exclusive-ored with bits of the group's number (16-byte words stay whole: the flush reads them).
constexpr int kBigPerThread = 1;
template <typename V> constexpr int kBigUnroll = 8 / sizeof(V);  // windows of 32 products a warp has in flight
// Default: three blocks of 384 threads per SM, so that two blocks sum while one looks for its pieces or flushes.  R-MAT
// scale 19 fp32 / block-dense fp32, ms of this kernel: 2 x 512 threads 24.1 / 8.0, 3 x 512 24.0 / 7.6, 3 x 256 23.9 / 8.6,
// 3 x 384 with four windows in flight 24.3 / 8.0, with two 22.9 / 7.2.  What binds it is the shared-memory pipe (70 % busy;
// the compare-and-swap of an add takes about eleven of its cycles per 32 products).
constexpr int kBigThreads = 384, kBigBlocks = 3;


template <typename V>
inline size_t big_task_smem_bytes(int W, int threads) {
  const size_t cap = static_cast<size_t>(threads) * kBigPerThread;
  return static_cast<size_t>(W) * sizeof(V) + cap * (sizeof(V) + 8) + 33 * 4 + 64;
}

template <typename V>
__device__ __forceinline__ u32 group_xor(u32 group) { return (group ^ (group >> 5)) & (32u - 16u / sizeof(V)); }
template <typename V>
__device__ __forceinline__ u32 big_slot(u32 c, u32 mask) { return (c & mask) ^ group_xor<V>(c >> 5); }
__device__ __forceinline__ float product(float a, float b) { return plus_zero(__fmul_rn(a, b)); }
__device__ __forceinline__ double product(double a, double b) { return plus_zero(__dmul_rn(a, b)); }

// slots of a 16-byte word of the accumulator that received something
__device__ __forceinline__ u32 touched_in(const int4& x, float) {
  constexpr int kIdle = static_cast<int>(0x80000000u);
  return (x.x != kIdle) + (x.y != kIdle) + (x.z != kIdle) + (x.w != kIdle);
}
__device__ __forceinline__ u32 touched_in(const int4& x, double) {
  constexpr int kIdle = static_cast<int>(0x80000000u);
  return (x.x != 0 || x.y != kIdle) + (x.z != 0 || x.w != kIdle);
}

template <typename V, int BT, int BLOCKS>
__global__ void __launch_bounds__(BT, BLOCKS) k6_big_tasks(
    TaskInput<V> in, const HeavyTask* __restrict__ tasks, i64 n_tasks, const int32_t* __restrict__ list, const int* __restrict__ counters,
    int* ticket, int32_t* __restrict__ out_col, V* __restrict__ out_val, u32* __restrict__ task_nnz) {
  extern __shared__ __align__(128) unsigned char smem_acc_raw[];
  constexpr int CAP = BT * kBigPerThread, PER = kBigPerThread, U = kBigUnroll<V>;
  constexpr int kWarps = BT / 32;
  const int W = 1 << in.log2_g;
  const u32 mask = static_cast<u32>(W - 1);
  V* acc = reinterpret_cast<V*>(smem_acc_raw);
  Pieces<V, CAP>& pc = *reinterpret_cast<Pieces<V, CAP>*>(smem_acc_raw + static_cast<size_t>(W) * sizeof(V));
  __shared__ uint2 s_sum[kWarps];
  __shared__ u32 s_scan[kWarps];
  __shared__ HeavyTask s_task[2];
  __shared__ int s_id[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const V idle = acc_idle(V(0));

  for (int s = tid; s < W; s += BT) acc[s] = idle;
  TaskFeed feed{ticket, counters[2] + counters[3], counters[2], list, n_tasks - 1, tasks};
  if (tid == 0) feed.start(&s_id[0], &s_task[0]);
  __syncthreads();
  int par = 0;
  int id = s_id[0];
  HeavyTask task = s_task[0];
  PieceRegs<V, PER> regs;
  if (id >= 0) {
    load_rows<V, BT, PER>(in, task, 0, regs);
    load_pieces<V, PER>(in, task, regs);
  }
  auto add = [&](u32 c, V v) { atomicAdd(&acc[big_slot<V>(c, mask)], v); };

  while (id >= 0) {
    if (tid == 0) feed.issue();
    // ---- accumulate, CAP rows of B at a time
    for (u32 r = 0;;) {
      const RoundSize rs = build_pieces<V, BT, PER>(regs, pc, s_sum);
      const bool more = ++r * static_cast<u32>(CAP) < task.n_a;
      if (more) load_rows<V, BT, PER>(in, task, r, regs);
      u32 c[U];
      V v[U], av[U];
      walk_products<V, CAP, U>(
          pc, rs, warp, kWarps,
          [&](int u, u32 src, V a) {
            c[u] = static_cast<u32>(in.b_col[src]);
            v[u] = in.b_val[src];
            av[u] = a;
          },
          [&](int u, bool valid, int) { if (valid) add(c[u], product(av[u], v[u])); });
      if (!more) break;
      load_pieces<V, PER>(in, task, regs);
      __syncthreads();
    }
    // ---- complete: flush.  The task's groups of 32 columns, an equal run of them per warp
    const u32 first_col = task.lo & ~mask;
    const int g_begin = static_cast<int>((task.lo & mask) >> 5), g_end = static_cast<int>((task.hi - first_col + 31) >> 5);
    const int per_warp = (g_end - g_begin + kWarps - 1) / kWarps;
    const int g0 = g_begin + warp * per_warp, g1 = min(g_end, g0 + per_warp);
    __syncthreads();
    if (tid == 0) feed.publish(&s_id[par ^ 1], &s_task[par ^ 1]);  // read after the next barrier
    u32 count = 0;
    {
      constexpr int kVec = 16 / sizeof(V);  // (a group is a whole number of 16-byte words, in whatever order its columns lie)
      const int4* const p = reinterpret_cast<const int4*>(acc);
#pragma unroll 4
      for (int i = g0 * (32 / kVec) + lane; i < g1 * (32 / kVec); i += 32) count += touched_in(p[i], V(0));
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0) s_scan[warp] = count;
    __syncthreads();
    const u32 wsum = lane < kWarps ? s_scan[lane] : 0u;
    const u32 total = __reduce_add_sync(0xffffffffu, wsum);
    u32 at = __reduce_add_sync(0xffffffffu, lane < warp ? wsum : 0u);
    if (tid == 0) task_nnz[id] = total;
    // the next task's first rows of B are requested before this task is written out
    const int next_id = s_id[par ^ 1];
    const HeavyTask next = s_task[par ^ 1];
    if (next_id >= 0) load_rows<V, BT, PER>(in, next, 0, regs);
    if (count) {
      constexpr int kVec = 16 / sizeof(V);
      int32_t* const c_col = out_col + task.off;
      V* const c_val = out_val + task.off;
      int4* const words = reinterpret_cast<int4*>(acc);
      for (int w = g0 * (32 / kVec) + lane; w - lane < g1 * (32 / kVec); w += 32) {
        // lane by lane in column order: the lane's word lies elsewhere inside its group
        const u32 g = static_cast<u32>(w) / (32 / kVec);
        const int at_w = w ^ static_cast<int>(group_xor<V>((first_col >> 5) + g) / kVec);
        const bool inside = w < g1 * (32 / kVec);
        V x[kVec];
        if (inside) *reinterpret_cast<int4*>(x) = words[at_w];
        bool some[kVec];
        u32 p = at, n = 0;
#pragma unroll
        for (int i = 0; i < kVec; ++i) {
          some[i] = inside && acc_touched(x[i]);
          const u32 m = __ballot_sync(0xffffffffu, some[i]);
          p += __popc(m & lanemask_lt());
          n += __popc(m);
        }
        at += n;
        if (n == 0) continue;
        int32_t col = static_cast<int32_t>(first_col) + w * kVec;
#pragma unroll
        for (int i = 0; i < kVec; ++i) {
          if (some[i]) {
            c_col[p] = col + i;
            c_val[p] = x[i];
            ++p;
          }
          x[i] = idle;
        }
        if (inside) words[at_w] = *reinterpret_cast<const int4*>(x);
      }
    }
    if (next_id >= 0) load_pieces<V, PER>(in, next, regs);
    __syncthreads();
    task = next;
    id = next_id;
    par ^= 1;
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// assembly
// ---------------------------------------------------------------------------------------------------------------------
// Entries per heavy row of the batch, from the prefix sums of the tasks' entries; heavy_total += the batch's entries.
__global__ void k_task_row_counts(const i64* __restrict__ nnz_off, const i64* __restrict__ row_task_off, i64 h0, i64 h1,
                                  const int32_t* __restrict__ x_heavy, int32_t* __restrict__ row_nnz, i64* __restrict__ heavy_total) {
  const i64 t0 = row_task_off[h0];
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(reinterpret_cast<u64*>(heavy_total), static_cast<u64>(nnz_off[row_task_off[h1] - t0]));
  for (i64 h = h0 + static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; h < h1; h += static_cast<i64>(gridDim.x) * blockDim.x)
    row_nnz[x_heavy[h]] = static_cast<int32_t>(nnz_off[row_task_off[h + 1] - t0] - nnz_off[row_task_off[h] - t0]);
}

// Position in C of every task's first entry, once C.rowPtr of the batch's rows is known (a thread per row).
__global__ void k_task_bases(const i64* __restrict__ nnz_off, const i64* __restrict__ row_task_off, i64 h0, i64 h1,
                             const int32_t* __restrict__ x_heavy, const i64* __restrict__ c_row_ptr, i64* __restrict__ base) {
  const i64 t0 = row_task_off[h0];
  for (i64 h = h0 + static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; h < h1; h += static_cast<i64>(gridDim.x) * blockDim.x) {
    const i64 a = row_task_off[h] - t0, b = row_task_off[h + 1] - t0;
    const i64 shift = c_row_ptr[x_heavy[h]] - nnz_off[a];
    for (i64 t = a; t < b; ++t) base[t] = nnz_off[t] + shift;
  }
}

// Everything between the sums and the gather in one launch of one block, for small products: prefix sums of the tasks'
// entries, entries per heavy row, C.rowPtr, position in C of every task's first entry, the gather's tile records, and the
// totals for the host.  (Five launches and a copy otherwise, each of which costs more than its work: 55 us from the last
// sum to the end of the call for R-MAT scales 10 to 12, of 130 to 260.)
constexpr int kTailWords = 10;  // totals the host reads at the end of an execute (see gm_plan::c_total)
constexpr i64 kFinishMax = 16384;  // tasks, and rows of A: above, one block takes as long as the launches
constexpr int kFinishThreads = 1024;
// out[0 .. n) = exclusive prefix sums of in (values from position n_valid on count as zero); returns the total (every thread).
// Ends with a barrier.
__device__ __forceinline__ i64 finish_scan(const u32* in, i64 n_valid, i64 n, i64* out, i64* tmp) {
  i64 run = 0;
  for (i64 i0 = 0; i0 < n; i0 += 4 * kFinishThreads) {
    const i64 i = i0 + threadIdx.x * 4;
    i64 v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = i + k < n_valid ? static_cast<i64>(in[i + k]) : 0;
      sum += v[k];
    }
    __syncthreads();
    i64 total;
    i64 ex = run + block_exclusive_scan(sum, tmp, &total);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i + k < n) out[i + k] = ex;
      ex += v[k];
    }
    run += total;
  }
  if (threadIdx.x == 0) out[n] = run;
  __syncthreads();
  return run;
}
__global__ void __launch_bounds__(kFinishThreads) k_finish_small(const u32* task_nnz, i64 n_tasks, i64* nnz_off, const i64* row_task_off,
                                                                 i64 n_heavy, const int32_t* x_heavy, int32_t* row_nnz, i64 n_rows,
                                                                 i64* c_row_ptr, i64* host_total, i64* base, int tile, TileMeta* meta,
                                                                 i64* totals, i64* host_totals) {
  __shared__ i64 tmp[33];
  const i64 heavy = finish_scan(task_nnz, row_task_off[n_heavy], n_tasks, nnz_off, tmp);  // (n_tasks: an upper bound)
  for (i64 h = threadIdx.x; h < n_heavy; h += kFinishThreads)
    row_nnz[x_heavy[h]] = static_cast<int32_t>(nnz_off[row_task_off[h + 1]] - nnz_off[row_task_off[h]]);
  __syncthreads();
  const i64 all = finish_scan(reinterpret_cast<const u32*>(row_nnz), n_rows, n_rows, c_row_ptr, tmp);
  for (i64 h = threadIdx.x; h < n_heavy; h += kFinishThreads) {
    const i64 a = row_task_off[h], b = row_task_off[h + 1];
    const i64 shift = c_row_ptr[x_heavy[h]] - nnz_off[a];
    for (i64 t = a; t < b; ++t) base[t] = nnz_off[t] + shift;
  }
  for (i64 t = threadIdx.x; t * tile < heavy; t += kFinishThreads) meta[t] = tile_bounds(nnz_off, n_tasks, 0, heavy, tile, t);
  if (threadIdx.x < kTailWords) host_totals[threadIdx.x] = threadIdx.x == 1 ? heavy : totals[threadIdx.x];
  if (threadIdx.x == 0) *host_total = all;  // (the host reads after a synchronisation)
}

// The plan's side of small products: tasks per row, their prefix sums and the tasks themselves in one launch of one block.
// The tables have room for an upper bound, so the host does not wait for the number of tasks.
// (Zipf-like, 4096 rows: 319 us with a count, a wait and an allocation in between, 284 with this.)
__global__ void __launch_bounds__(kFinishThreads) k_plan_small(const u32* counts, const i64* heavy_base, i64 n_heavy, TaskRules r,
                                                               u32* row_tasks, i64* row_task_off, const int32_t* x_heavy,
                                                               const i64* a_row_ptr, const u32* parts_tab, TaskTables tt,
                                                               const unsigned char* in_panel) {
  __shared__ i64 tmp[33];
  for (i64 h = threadIdx.x; h < n_heavy; h += kFinishThreads)
    row_tasks[h] = in_panel && in_panel[h] ? 1 : cut_row(counts + h * r.granules, static_cast<u32>(heavy_base[h + 1] - heavy_base[h]), r, [](int, int, u32, u32) {});
  __syncthreads();
  finish_scan(row_tasks, n_heavy, n_heavy, row_task_off, tmp);
  __shared__ u32 s_n[4];
  if (threadIdx.x < 4) s_n[threadIdx.x] = 0u;
  __syncthreads();
  for (i64 h = threadIdx.x; h < n_heavy; h += kFinishThreads)
    emit_row(counts, heavy_base, h, 0, r, row_task_off[h], x_heavy, a_row_ptr, parts_tab, tt, in_panel,
             [&](int c) { return atomicAdd(&s_n[c], 1u); });
  __syncthreads();
  if (threadIdx.x < 4) tt.counters[threadIdx.x] = static_cast<int>(s_n[threadIdx.x]);
}

}  // namespace gm
