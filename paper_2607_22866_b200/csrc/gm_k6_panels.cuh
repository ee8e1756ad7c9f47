// K6p — panels: neighbouring heavy rows of A with much the same columns (dense blocks of structural matrices, several
// unknowns per node) are summed together.
//
// Row by row, such rows walk the same rows of B again and again, and every product is an add in shared memory.  A panel of up
// to 32 rows is a small dense matrix instead: its columns are the union U of the rows' columns, and the rows of B in U,
// spread out over groups of neighbouring columns, are the other factor.  Both are brought in once per panel and multiplied in registers.
//   plan     k_panel_similar  does a heavy row share half of its columns with the one before (32 samples)
//            k_panel_cut      runs of similar rows, cut into panels
//            k_piece_count, k_piece_fill  the pieces of every row of B per group of neighbouring columns
//            k_panel_build    U with a mask of the rows that hold each column; per group of columns of C the pieces of rows of B
//                             that reach it (visits), and where the group's entries of every row go; kept if it pays
//   execute  k6_panels        a warp per group, a unit of eight or sixteen groups of a panel to a block
// A panel's row is one task (see gm_k6_tasks.cuh) that is in no list: its entries go to the row's place in the staging area.
//
// What bounds it: nothing near its limit; block-dense fp32, 1.3 G products in 0.53 ms, issue slots 42 % with sixteen warps per SM (two blocks
// of 128 registers a thread), which wait for the next visits' entries and, at the end of a panel, for one another.  A product costs five
// warp instructions per 32, against 135 by the dense accumulator, whose kernel took 5.7 + 1.4 ms of the call's 8.5 for 2.7 G products;
// now 1.03 ms, the lists 0.30 ms, the call 2.35.
#pragma once
#include "gm_common.cuh"
#include "gm_k6_tasks.cuh"

namespace gm {

constexpr int kPanelRows = 32;
constexpr int kPanelMinRows = 2;
constexpr int kPanelThreads = 256, kPanelWarps = kPanelThreads / 32;
constexpr int kPanelMaxGroups = 16384;                      // of C
constexpr int kPanelMaxReach = 512;                         // groups that a panel reaches
constexpr i64 kPanelMaxRowsB = i64{1} << 19;                // (the bitmap of a panel's columns is in shared memory)
// Columns of a panel: with its part of A in shared memory two blocks fit an SM.
constexpr int kPanelMaxU = 704;
template <typename V> constexpr int kPanelColumns = sizeof(V) == 4 ? kPanelMaxU : 384;
// Columns of a group: what a warp multiplies at a time.
template <typename V> constexpr int kPanelGroup = 256 / sizeof(V);
inline int panel_group_bits(int val_bytes) { return val_bytes == 4 ? 6 : 5; }
// What panels cost, counted in products of the dense accumulator, which has `piece` of them to add for every entry of A.  A unit takes a
// block some 15 us, and a warp 0.3 us for each visit of its groups, whether two rows are in it or thirty-two.  (fp32: 1.7 ps a product and
// 115 a piece against 0.07 us a unit and 1.05 ns a visit of all eight warps, with 296 blocks at a time; fp64 2.9 ps and 100 against 0.07 and 1.1.)
// 16000 rows in groups of R alike, 80 to 95 entries each, rows of B with k entries in n columns, us a call by tasks / by panels, fp32:
//   R 2, k 150, n 200    712 / 1523    R 4, k 200, n 300  833 / 966    R 8, k 150, n 500    699 / 670    R 32, k 150, n 2000  883 / 826
//   R 3, k 100, n 300    606 / 1211    R 4, k 200, n 230  832 / 907    R 16, k 150, n 1500  810 / 928    R 32, k 150, n 1500  812 / 679
//   R 4, k 200, n 400    842 / 1035    R 8, k 150, n 700  736 / 942    R 16, k 150, n 800   745 / 687    (panels from R 8, n 500 on but R 16, n 1500)
// fp64: R 4, k 200, n 300 and 230  1031 / 1288, 1016 / 922; R 8, n 400, k 100 and 150  711 / 842, 853 / 843 (panels for the second of both).
struct PanelCost {
  float piece, unit, visit;
};
template <typename V> constexpr PanelCost kPanelCost = sizeof(V) == 4 ? PanelCost{66.f, 41000.f, 610.f} : PanelCost{35.f, 24500.f, 380.f};
// Once there are lists, panels with fewer products per visit than this stay with the tasks.
constexpr u32 kPanelMinProducts = 40;
// Room for pieces of rows of B, per entry of B, and for visits and groups, per entry of A in panels; what takes more is left to the tasks.
constexpr int kPanelEntriesPerPiece = 4, kPanelVisitsPerEntry = 3, kPanelEntriesPerGroup = 8;

struct Panel {
  u32 h, rows, n_u, n_groups;  // first heavy row, rows, columns of U, groups reached (n_u = 0: not a panel)
  i64 e;                       // entries of A in the panels before
};
struct __align__(16) GroupPiece {  // the entries of a row of B in one group
  u32 start;      // position of the first in B's arrays
  u32 group;
  u64 mask;       // their columns
};
struct PanelGroup {
  u32 group, first, n;  // which, its visits (relative to the panel's)
};
struct PanelVisit {
  u32 piece, u;   // a piece of the row of B that column u of U selects
};
struct PanelUnit {
  u32 panel, group, n;  // n groups from this one
};
struct PanelTables {
  i64* piece_ptr;         // per row of B: its first piece
  GroupPiece* pieces;
  i64 max_pieces;
  Panel* list;
  u64* counts;            // kPanelCounts: see below
  unsigned char* of_row;  // per heavy row: 1 = in a panel
  PanelUnit* units;
  // of a panel: from its e (a_u, u_mask), e * kPanelVisitsPerEntry (visits) and e / kPanelEntriesPerGroup (groups) on
  unsigned short* a_u;    // the entry's column in U
  u32* u_mask;
  PanelVisit* visits;
  PanelGroup* groups;
  u32* group_rows;        // per group and row: entries of the row in the panel's groups before; behind the last group: in all
};

// Pieces per row of B; a warp per row.
__global__ void __launch_bounds__(256) k_piece_count(const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, i64 n_rows_b,
                                                     int group_bits, u32* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  for (i64 k = static_cast<i64>(blockIdx.x) * 8 + (threadIdx.x >> 5); k < n_rows_b; k += static_cast<i64>(gridDim.x) * 8) {
    const i64 s = b_row_ptr[k], e = b_row_ptr[k + 1];
    u32 n = 0;
#pragma unroll 4
    for (i64 i = s + lane; i < e; i += 32) n += i == s || (b_col[i] >> group_bits) != (b_col[i - 1] >> group_bits);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) count[k] = n;
  }
}
// Panels take the order of their rows from the matrices' contract and look whether it holds, since the tasks, with columns that fit one
// granule, give the right sums without it: there are no panels where a row of B is not strictly ascending, and a row of A that is
// not leaves its panel to the tasks.
__global__ void __launch_bounds__(256) k_piece_fill(const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, i64 n_rows_b,
                                                    int group_bits, PanelTables pt) {
  if (pt.piece_ptr[n_rows_b] > pt.max_pieces) return;
  const int lane = threadIdx.x & 31;
  bool bad = false;
  for (i64 k = static_cast<i64>(blockIdx.x) * 8 + (threadIdx.x >> 5); k < n_rows_b; k += static_cast<i64>(gridDim.x) * 8) {
    const i64 s = b_row_ptr[k], e = b_row_ptr[k + 1];
    GroupPiece* const out = pt.pieces + pt.piece_ptr[k];
    int n = 0;
    for (i64 i0 = s; i0 < e; i0 += 32) {
      const i64 i = i0 + lane;
      const int32_t c = i < e ? b_col[i] : INT_MAX, before = i < e && i > s ? b_col[i - 1] : -1;
      const int g = c >> group_bits;
      const bool head = i < e && (i == s || (before >> group_bits) != g);
      bad |= c <= before;
      const u32 heads = __ballot_sync(0xffffffffu, head);
      if (head) {
        const int at = n + __popc(heads & lanemask_lt());
        out[at].start = static_cast<u32>(i);
        out[at].group = static_cast<u32>(g);
      }
      n += __popc(heads);
    }
    __syncwarp();
    for (int q = lane; q < n; q += 32) {  // a lane per piece
      const volatile GroupPiece* const v = out;
      const u32 first = v[q].start, last = q + 1 < n ? v[q + 1].start : static_cast<u32>(e);
      u64 m = 0;
#pragma unroll 4
      for (u32 i = first; i < last; ++i) m |= 1ull << (b_col[i] & ((1 << group_bits) - 1));
      out[q].mask = m;
    }
    __syncwarp();
  }
  if (bad) pt.counts[kPanelUnordered] = 1ull;
}

// A warp per heavy row: similar[h] = 1 if about half of the row's columns are in heavy row h - 1, and neither is much longer.
// Some of those rows, spread out, are looked at closer: how many columns they share, and how many pieces a row of B that they use has.
constexpr i64 kPanelSampleAll = 1024;  // heavy rows up to which all are, and about one in 32 above
__global__ void __launch_bounds__(256) k_panel_similar(const int32_t* __restrict__ x_heavy, i64 n_heavy, const i64* __restrict__ a_row_ptr,
                                                       const int32_t* __restrict__ a_col, const i64* __restrict__ b_row_ptr,
                                                       const int32_t* __restrict__ b_col, int group_bits, u64* __restrict__ counts,
                                                       unsigned char* __restrict__ similar) {
  const i64 h = static_cast<i64>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (h >= n_heavy) return;
  const int lane = threadIdx.x & 31;
  bool hit = false;
  i64 n = 0, n0 = 0, s = 0;
  if (h > 0) {
    const i64 row = x_heavy[h], prev = x_heavy[h - 1];
    s = a_row_ptr[row];
    const i64 s0 = a_row_ptr[prev];
    n = a_row_ptr[row + 1] - s;
    n0 = a_row_ptr[prev + 1] - s0;
    const i64 j = n <= 32 ? lane : n * lane / 32;
    if (j < n) {
      const int32_t c = a_col[s + j];
      i64 lo = 0, hi = n0;
      while (lo < hi) {
        const i64 mid = (lo + hi) >> 1;
        if (a_col[s0 + mid] < c) lo = mid + 1; else hi = mid;
      }
      hit = lo < n0 && a_col[s0 + lo] == c;
    }
  }
  const int hits = __popc(__ballot_sync(0xffffffffu, hit));
  const int tried = static_cast<int>(min(n, i64{32}));
  const bool alike = hits > 0 && hits * 9 >= tried * 4 && 2 * min(n, n0) >= max(n, n0);
  if (lane == 0) similar[h] = alike;
  const u32 mix = static_cast<u32>(h) * 2654435761u;
  if (!alike || (n_heavy > kPanelSampleAll && mix >> 27 != 0)) return;
  const int32_t k = a_col[s + (mix >> 3) % n];
  const i64 b0 = b_row_ptr[k], b1 = b_row_ptr[k + 1];
  u32 pieces = 0;
  for (i64 i = b0 + lane; i < b1; i += 32) pieces += i == b0 || (b_col[i] >> group_bits) != (b_col[i - 1] >> group_bits);
  pieces = __reduce_add_sync(0xffffffffu, pieces);
  if (lane == 0) {
    atomicAdd(&counts[kPanelTried], static_cast<u64>(tried));
    atomicAdd(&counts[kPanelHits], static_cast<u64>(hits));
    atomicAdd(&counts[kPanelSampled], 1ull);
    atomicAdd(&counts[kPanelPieces], static_cast<u64>(pieces));
    atomicAdd(&counts[kPanelSampleLen], static_cast<u64>(b1 - b0));
  }
}

// A block per 1024 heavy rows (runs end there, and where a batch begins).  starts: first rows of the batches.
__global__ void __launch_bounds__(1024) k_panel_cut(const unsigned char* __restrict__ similar, i64 n_heavy, const i64* __restrict__ starts,
                                                    int n_batches, const i64* __restrict__ heavy_base, const i64* __restrict__ heavy_nz_off,
                                                    int n_groups, int unit_groups, PanelCost cost, PanelTables pt, u64* __restrict__ host_counts) {
  __shared__ int s_first[1024], s_end[1024];
  const int tid = threadIdx.x;
  const i64 h = static_cast<i64>(blockIdx.x) * 1024 + tid;
  const int n = static_cast<int>(min(i64{1024}, n_heavy - static_cast<i64>(blockIdx.x) * 1024));
  bool first = tid == 0 || h >= n_heavy || !similar[h];
  for (int lo = 0, hi = n_batches; lo < hi && !first;) {
    const int mid = (lo + hi) >> 1;
    if (starts[mid] == h) first = true;
    else if (starts[mid] < h) lo = mid + 1; else hi = mid;
  }
  s_first[tid] = first ? tid : 0;
  s_end[tid] = first ? tid : n;  // of the run before
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int a = tid >= o ? s_first[tid - o] : 0;
    const int b = tid + o < 1024 ? s_end[tid + o] : n;
    __syncthreads();
    s_first[tid] = max(s_first[tid], a);
    s_end[tid] = min(s_end[tid], b);
    __syncthreads();
  }
  if (h < n_heavy) {
    pt.of_row[h] = 0;
    const int begin = s_first[tid], end = min(tid + 1 < 1024 ? s_end[tid + 1] : n, n);
    const int len = end - begin, pieces = (len + kPanelRows - 1) / kPanelRows, per = (len + pieces - 1) / pieces;
    const int rows = (tid - begin) % per ? 0 : min(per, end - tid);
    if (rows >= kPanelMinRows) {
      const u64 at = atomicAdd(&pt.counts[kPanelsFound], 1ull);
      const i64 entries = heavy_nz_off[h + rows] - heavy_nz_off[h];
      const u64 e = atomicAdd(&pt.counts[kPanelEntries], static_cast<u64>(entries));
      // what the panel is expected to gain: its columns by what neighbouring rows share, its visits by the pieces of some rows of B
      const float pieces = static_cast<float>(pt.counts[kPanelPieces]) / fmaxf(1.f, static_cast<float>(pt.counts[kPanelSampled]));
      const float share = static_cast<float>(pt.counts[kPanelHits]) / fmaxf(1.f, static_cast<float>(pt.counts[kPanelTried]));
      const float visits = static_cast<float>(entries) / static_cast<float>(rows) / fmaxf(share, 0.25f) * pieces;
      // (with 10 % more than there is room for, which is counted when the lists are built; nothing where no row was looked at closer)
      const bool room = pt.counts[kPanelSampled] != 0 && pieces * (kPanelEntriesPerPiece * 0.9f) <= static_cast<float>(pt.counts[kPanelSampleLen]) / fmaxf(1.f, static_cast<float>(pt.counts[kPanelSampled])) &&
                        visits * 0.9f <= static_cast<float>(entries) * kPanelVisitsPerEntry;
      const float by_tasks = static_cast<float>(heavy_base[h + rows] - heavy_base[h]) + cost.piece * static_cast<float>(entries);
      const float by_panel = cost.unit * ceilf(pieces / static_cast<float>(unit_groups)) + cost.visit * visits / static_cast<float>(min(n_groups, kPanelWarps));
      const float gain = room ? by_tasks - by_panel : fminf(by_tasks - by_panel, 0.f);
      atomicAdd(&pt.counts[kPanelGain], static_cast<u64>(static_cast<i64>(gain)));  // (of either sign)
      pt.list[at] = Panel{static_cast<u32>(h), static_cast<u32>(rows), 0u, 0u, static_cast<i64>(e)};
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0 && atomicAdd(&pt.counts[kPanelBlocks], 1ull) == gridDim.x - 1) {  // the last block: the counts to the host
    __threadfence();
    for (int i = 0; i < kPanelCounts; ++i) host_counts[i] = static_cast<const volatile u64*>(pt.counts)[i];  // (read after an event)
  }
}

constexpr int kPanelBuildThreads = 512;
struct PanelBuildSmem {
  u32 mask[kPanelMaxU];
  int32_t u_col[kPanelMaxU];
  u32 first[kPanelMaxReach + 1];       // visits of the groups before
  unsigned short group[kPanelMaxReach];
  unsigned short n_rows[kPanelMaxReach][kPanelRows];  // entries of a row in a group
  i64 row[kPanelRows];
  i64 off[kPanelRows + 1];             // a row's first entry in the lists
  int n[kPanelRows];
  int lo, hi, tmp[33];
  i64 tmp64[33];
};
// columns of A: bitmap and ranks; groups of C: visits, then cursors
inline size_t panel_build_smem(i64 n_rows_b, i64 n_groups) {
  return sizeof(PanelBuildSmem) + static_cast<size_t>((n_rows_b + 31) / 32) * 6 + static_cast<size_t>(n_groups) * 4 + 64;
}
// A block per panel.  max_u: columns of a panel that fit the product's shared memory.  unit_groups: groups of a unit.
__global__ void __launch_bounds__(kPanelBuildThreads) k_panel_build(
    PanelTables pt, const int32_t* __restrict__ x_heavy, const i64* __restrict__ heavy_base, const i64* __restrict__ heavy_nz_off,
    const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col, i64 n_rows_b, int n_groups, int max_u, int unit_groups) {
  extern __shared__ __align__(16) unsigned char smem_build_raw[];
  constexpr int T = kPanelBuildThreads, kWarps = T / 32;
  PanelBuildSmem& sm = *reinterpret_cast<PanelBuildSmem*>(smem_build_raw);
  const int n_words_max = static_cast<int>((n_rows_b + 31) / 32);
  u32* const bits = reinterpret_cast<u32*>(smem_build_raw + ((sizeof(PanelBuildSmem) + 15) & ~size_t{15}));
  u32* const g_count = bits + n_words_max;
  unsigned short* const before = reinterpret_cast<unsigned short*>(g_count + n_groups);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 n_panels = pt.piece_ptr[n_rows_b] > pt.max_pieces || pt.counts[kPanelUnordered] ? 0u : static_cast<u32>(pt.counts[kPanelsFound]);
  for (u32 q = blockIdx.x; q < n_panels; q += gridDim.x) {
    const Panel p = pt.list[q];
    const int R = static_cast<int>(p.rows);
    __syncthreads();
    if (tid == 0) { sm.lo = INT_MAX; sm.hi = 0; }
    __syncthreads();
    if (tid >= 64 && tid <= 64 + R) sm.off[tid - 64] = p.e + (heavy_nz_off[p.h + tid - 64] - heavy_nz_off[p.h]);
    if (tid < R) {
      const i64 row = x_heavy[p.h + tid];
      const i64 s = a_row_ptr[row];
      const int n = static_cast<int>(a_row_ptr[row + 1] - s);  // (a heavy row has entries)
      sm.row[tid] = s;
      sm.n[tid] = n;
      atomicMin(&sm.lo, a_col[s] >> 5);
      atomicMax(&sm.hi, a_col[s + n - 1] >> 5);
    }
    __syncthreads();
    // ---- U: the columns as a bitmap, their ranks, the rows that hold them
    const int w0 = sm.lo, n_words = max(sm.hi - sm.lo, 0) + 1;
    for (int w = tid; w < n_words; w += T) bits[w] = 0u;
    for (int i = tid; i < kPanelMaxU; i += T) sm.mask[i] = 0u;
    for (int g = tid; g < n_groups; g += T) g_count[g] = 0u;
    __syncthreads();
    bool bad = false;  // not ascending: a column outside the range of the rows' ends
    for (int r = warp; r < R; r += kWarps) {
#pragma unroll 4
      for (int j = lane; j < sm.n[r]; j += 32) {
        const int c = a_col[sm.row[r] + j];
        const u32 bit = 1u << (c & 31);
        const u32 at = static_cast<u32>((c >> 5) - w0), w = min(at, static_cast<u32>(n_words - 1));
        bad |= at != w;
        if (!(bits[w] & bit)) atomicOr(&bits[w], bit);
      }
    }
    if (__syncthreads_or(bad)) continue;  // (block-uniform, as all that follow)
    int n_u = 0;
    for (int i0 = 0; i0 < n_words; i0 += T) {
      const int w = i0 + tid;
      const int n = w < n_words ? __popc(bits[w]) : 0;
      int total;
      const int ex = block_exclusive_scan(n, sm.tmp, &total);
      if (w < n_words) before[w] = static_cast<unsigned short>(min(n_u + ex, 0xffff));
      n_u += total;
      __syncthreads();
    }
    if (n_u > max_u) continue;
    for (int r = warp; r < R; r += kWarps) {
      const i64 at = sm.off[r];
#pragma unroll 4
      for (int j = lane; j < sm.n[r]; j += 32) {
        const int c = a_col[sm.row[r] + j];
        const int w = (c >> 5) - w0;
        const int u = before[w] + __popc(bits[w] & ((1u << (c & 31)) - 1u));
        atomicOr(&sm.mask[u], 1u << r);
        pt.a_u[at + j] = static_cast<unsigned short>(u);
      }
    }
    for (int w = tid; w < n_words; w += T) {
      int u = before[w];
      for (u32 b = bits[w]; b; b &= b - 1, ++u) sm.u_col[u] = (w0 + w) * 32 + __ffs(b) - 1;
    }
    __syncthreads();
    // ---- visits per group
    i64 mine = 0;  // (visits << 32) | entries in the masks, fewer than in the rows where a row has a column twice
    for (int u = tid; u < n_u; u += T) {
      const i64 s = pt.piece_ptr[sm.u_col[u]], e = pt.piece_ptr[sm.u_col[u] + 1];
#pragma unroll 4
      for (i64 i = s; i < e; ++i) atomicAdd(&g_count[pt.pieces[i].group], 1u);
      mine += ((e - s) << 32) + __popc(sm.mask[u]);
    }
    i64 sums;
    block_exclusive_scan(mine, sm.tmp64, &sums);
    const i64 n_visits = sums >> 32;
    const i64 entry0 = sm.off[0], entries = sm.off[R] - entry0;
    const i64 products = heavy_base[p.h + R] - heavy_base[p.h];
    if ((sums & 0xffffffff) != entries || products < n_visits * kPanelMinProducts || n_visits > entries * kPanelVisitsPerEntry) continue;
    __syncthreads();
    int n_g = 0, run = 0;
    for (int i0 = 0; i0 < n_groups; i0 += T) {
      const int g = i0 + tid;
      const int n = g < n_groups ? static_cast<int>(g_count[g]) : 0;
      int total, some;
      const int at = block_exclusive_scan(n, sm.tmp, &total);
      __syncthreads();
      const int rank = n_g + block_exclusive_scan(n ? 1 : 0, sm.tmp, &some);
      __syncthreads();
      if (n && rank < kPanelMaxReach) {
        g_count[g] = static_cast<u32>(run + at);  // (from here on the group's next visit)
        sm.group[rank] = static_cast<unsigned short>(g);
        sm.first[rank] = static_cast<u32>(run + at);
      }
      n_g += some;
      run += total;
    }
    // (the last group's sums lie behind it)
    if (n_g + 1 > kPanelMaxReach || (n_g + 1) * kPanelEntriesPerGroup > entries) continue;
    const i64 visit0 = entry0 * kPanelVisitsPerEntry;
    if (tid == 0) sm.first[n_g] = static_cast<u32>(run);
    __syncthreads();
    for (int u = tid; u < n_u; u += T) {
      const i64 s = pt.piece_ptr[sm.u_col[u]], e = pt.piece_ptr[sm.u_col[u] + 1];
#pragma unroll 4
      for (i64 i = s; i < e; ++i)
        pt.visits[visit0 + atomicAdd(&g_count[pt.pieces[i].group], 1u)] = PanelVisit{static_cast<u32>(i), static_cast<u32>(u)};
    }
    __threadfence_block();
    __syncthreads();
    // ---- entries per row and group
    const i64 group0 = (entry0 + kPanelEntriesPerGroup - 1) / kPanelEntriesPerGroup;
    for (int k = warp; k < n_g; k += kWarps) {
      u32 rows0 = 0, rows1 = 0;
      const int first = static_cast<int>(sm.first[k]), last = static_cast<int>(sm.first[k + 1]);
      for (int i0 = first; i0 < last; i0 += 32) {  // 32 visits at once, a lane each
        u64 m = 0;
        u32 rows = 0;
        if (i0 + lane < last) {
          const PanelVisit v = pt.visits[visit0 + i0 + lane];
          m = pt.pieces[v.piece].mask;
          rows = sm.mask[v.u];
        }
        const u32 lo = static_cast<u32>(m), hi = static_cast<u32>(m >> 32);
        const int n = min(32, last - i0);
        for (int i = 0; i < n; ++i) {
          const u32 r = __shfl_sync(0xffffffffu, rows, i);
          if (__shfl_sync(0xffffffffu, lo, i) >> lane & 1u) rows0 |= r;
          if (__shfl_sync(0xffffffffu, hi, i) >> lane & 1u) rows1 |= r;
        }
      }
      u32 n = 0;
#pragma unroll 4
      for (int r = 0; r < kPanelRows; ++r) {
        const u32 c = __popc(__ballot_sync(0xffffffffu, rows0 >> r & 1u)) + __popc(__ballot_sync(0xffffffffu, rows1 >> r & 1u));
        if (lane == r) n = c;
      }
      sm.n_rows[k][lane] = static_cast<unsigned short>(n);
      if (lane == 0) pt.groups[group0 + k] = PanelGroup{static_cast<u32>(sm.group[k]), static_cast<u32>(first), static_cast<u32>(last - first)};
    }
    __syncthreads();
    if (warp == 0) {
      u32 n = 0;
#pragma unroll 4
      for (int k = 0; k < n_g; ++k) {
        pt.group_rows[(group0 + k) * kPanelRows + lane] = n;
        n += sm.n_rows[k][lane];
      }
      pt.group_rows[(group0 + n_g) * kPanelRows + lane] = n;
    }
    for (int u = tid; u < n_u; u += T) pt.u_mask[entry0 + u] = sm.mask[u];
    if (tid < R) pt.of_row[p.h + tid] = 1;
    if (tid == 0) {
      pt.list[q].n_u = static_cast<u32>(n_u);
      pt.list[q].n_groups = static_cast<u32>(n_g);
      const int n = (n_g + unit_groups - 1) / unit_groups;
      const u64 at = atomicAdd(&pt.counts[kPanelUnits], static_cast<u64>(n));
      for (int i = 0; i < n; ++i)
        pt.units[at + i] = PanelUnit{q, static_cast<u32>(i * unit_groups), static_cast<u32>(min(unit_groups, n_g - i * unit_groups))};
    }
  }
}

// Debug mode: the lists of every panel (a block each) hold its products and no others, in the columns and at the places that they say:
// entries of A find the column of U that selects their row of B; the visits are pieces of those rows, with the entries that their masks
// say, in the group that lists them; they add up to the products; the entries of a row fit its part of the staging area.
__global__ void __launch_bounds__(256) k_validate_panels(PanelTables pt, const int32_t* __restrict__ x_heavy, i64 n_heavy,
                                                         const i64* __restrict__ heavy_base, const i64* __restrict__ heavy_nz_off,
                                                         const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col,
                                                         const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, i64 n_rows_b,
                                                         i64 n_cols, int group_bits, int* __restrict__ err) {
  __shared__ int s_col[kPanelMaxU];
  __shared__ u32 s_mask[kPanelMaxU];
  __shared__ i64 s_sum[33];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (i64 q = blockIdx.x; q < static_cast<i64>(pt.counts[kPanelsFound]); q += gridDim.x) {
    const Panel p = pt.list[q];
    if (p.n_u == 0) continue;
    if (p.n_u > kPanelMaxU || p.n_groups >= kPanelMaxReach || p.rows > kPanelRows || static_cast<i64>(p.h) + p.rows > n_heavy) {
      if (tid == 0) dev_set_error(err, kDevBadChunk);
      continue;
    }
    const int R = static_cast<int>(p.rows);
    const i64 entries = heavy_nz_off[p.h + R] - heavy_nz_off[p.h], group0 = (p.e + kPanelEntriesPerGroup - 1) / kPanelEntriesPerGroup;
    bool bad = false;
    i64 bits = 0;
    for (int u = tid; u < static_cast<int>(p.n_u); u += 256) {
      s_col[u] = -1;
      s_mask[u] = pt.u_mask[p.e + u];
      bits += __popc(s_mask[u]);
    }
    __syncthreads();
    for (int r = warp; r < R; r += 8) {
      const i64 row = x_heavy[p.h + r], from = a_row_ptr[row], at = p.e + (heavy_nz_off[p.h + r] - heavy_nz_off[p.h]);
      for (i64 j = lane; j < a_row_ptr[row + 1] - from; j += 32) {
        const int k = a_col[from + j];
        const u32 u = pt.a_u[at + j];
        if (u >= p.n_u || k < 0 || k >= n_rows_b) {
          bad = true;
          continue;
        }
        const int was = atomicCAS(&s_col[u], -1, k);
        bad |= (was != -1 && was != k) || !(s_mask[u] >> r & 1u);
      }
    }
    i64 n;
    block_exclusive_scan(bits, s_sum, &n);
    bad |= n != entries;
    __syncthreads();
    i64 products = 0;
    for (int k = warp; k < static_cast<int>(p.n_groups); k += 8) {
      const PanelGroup g = pt.groups[group0 + k];
      if (static_cast<i64>(g.first) + g.n > entries * kPanelVisitsPerEntry) {
        bad = true;
        continue;
      }
      for (u32 i = lane; i < g.n; i += 32) {
        const PanelVisit v = pt.visits[p.e * kPanelVisitsPerEntry + g.first + i];
        const int row = v.u < p.n_u ? s_col[v.u] : -1;
        if (row < 0 || v.piece < pt.piece_ptr[row] || v.piece >= pt.piece_ptr[row + 1]) {
          bad = true;
          continue;
        }
        const GroupPiece piece = pt.pieces[v.piece];
        const int m = __popcll(piece.mask);
        bad |= piece.group != g.group;
        if (piece.start < b_row_ptr[row] || static_cast<i64>(piece.start) + m > b_row_ptr[row + 1]) {
          bad = true;
          continue;
        }
        u64 left = piece.mask;
        for (int t = 0; t < m; ++t, left &= left - 1) {
          const i64 c = b_col[piece.start + t];
          bad |= c >= n_cols || c != (static_cast<i64>(g.group) << group_bits) + __ffsll(static_cast<long long>(left)) - 1;
        }
        products += static_cast<i64>(m) * __popc(s_mask[v.u]);
      }
    }
    block_exclusive_scan(products, s_sum, &n);
    bad |= n != heavy_base[p.h + R] - heavy_base[p.h];
    if (tid < R) {
      u32 before = 0;
      for (u32 k = 0; k <= p.n_groups; ++k) {
        const u32 m = pt.group_rows[(group0 + k) * kPanelRows + tid];
        bad |= m < before || m - before > 1u << group_bits;
        before = m;
      }
      bad |= before > heavy_base[p.h + tid + 1] - heavy_base[p.h + tid];
    }
    if (bad) dev_set_error(err, kDevBadChunk);
    __syncthreads();  // (the arrays are the next panel's)
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// the product of a panel
// ---------------------------------------------------------------------------------------------------------------------
// The panel's part of A lies in shared memory as a dense matrix, a column of 32 rows per u.  A warp takes one group of columns of C at a
// time and goes over its visits, kPanelDepth together: their entries, spread out over the group's columns by their mask, to rows of the
// warp's own (the next ones' are on the way meanwhile), then a rank-1 update each: a lane has 8 rows x 8 columns (fp64: 8 x 4) of
// the sums in registers.
// Which of the entries exist follows from masks alone: column c of row r has one if some visit's u has both.
// What is not there counts as zero, which is right as long as all is finite: with an infinity or a NaN in the panel's A or in a
// round of visits the products are formed entry by entry instead.
constexpr int kPanelDepth = 4;
static_assert(kPanelDepth == 4 && 32 % kPanelDepth == 0, "entries leave four rows at a time through the visits' rows; a warp's 32 visits are whole rounds");
template <typename V>
struct PanelSmem {
  static constexpr int kStride = kPanelRows + 16 / sizeof(V);  // (columns of A are filled row by row: not all in one bank)
  V part[kPanelWarps][kPanelDepth][kPanelGroup<V>];
  V dense[kPanelColumns<V> * kStride];
  u32 u_mask[kPanelColumns<V>];
  i64 row_out[kPanelRows];  // place of the row in the staging area
  int ticket;
};
__device__ __forceinline__ bool finite_bits(float x) { return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u; }
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

template <typename V>
__global__ void __launch_bounds__(kPanelThreads, 2) k6_panels(
    const i64* __restrict__ a_row_ptr, const V* __restrict__ a_val, const V* __restrict__ b_val, PanelTables pt,
    const int32_t* __restrict__ x_heavy, const i64* __restrict__ heavy_base, const i64* __restrict__ heavy_nz_off, i64 h0, i64 h1, i64 elem0,
    const i64* __restrict__ row_task_off, int* __restrict__ ticket, int32_t* __restrict__ out_col, V* __restrict__ out_val,
    u32* __restrict__ task_nnz, u64* __restrict__ total_rows) {
  constexpr int G = kPanelGroup<V>, D = kPanelDepth, S = PanelSmem<V>::kStride;
  constexpr int CH = G / 32;           // 32-column halves of a group
  constexpr int CC = G / 8;            // columns of a lane
  constexpr int VEC = 16 / sizeof(V);  // they come in 16-byte runs: run i at i * 8 * VEC + cg * VEC
  extern __shared__ __align__(16) unsigned char smem_panel_raw[];
  PanelSmem<V>& sm = *reinterpret_cast<PanelSmem<V>*>(smem_panel_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = lane >> 3, cg = lane & 7;  // the lane's rows rg * 8 .. + 7
  const int n_units = static_cast<int>(pt.counts[kPanelUnits]);
  V(*const part)[G] = sm.part[warp];
  for (;;) {
    __syncthreads();
    if (tid == 0) sm.ticket = atomicAdd(ticket, 1);
    __syncthreads();
    if (sm.ticket >= n_units) return;
    const PanelUnit unit = pt.units[sm.ticket];
    const Panel p = pt.list[unit.panel];
    if (p.h < h0 || p.h >= h1) continue;
    const int n_u = static_cast<int>(p.n_u), R = static_cast<int>(p.rows);
    const i64 entry0 = p.e, group0 = (entry0 + kPanelEntriesPerGroup - 1) / kPanelEntriesPerGroup;
    // ---- the panel's part of A
    for (int i = tid; i < n_u * S / VEC; i += kPanelThreads) reinterpret_cast<int4*>(sm.dense)[i] = make_int4(0, 0, 0, 0);
    for (int u = tid; u < n_u; u += kPanelThreads) sm.u_mask[u] = pt.u_mask[entry0 + u];
    if (tid < kPanelRows) sm.row_out[tid] = tid < R ? heavy_base[p.h + tid] - elem0 : 0;
    __syncthreads();
    bool a_bad = false;
    for (int r = warp; r < R; r += kPanelWarps) {
      const i64 from = a_row_ptr[x_heavy[p.h + r]], before = heavy_nz_off[p.h + r], at = entry0 + (before - heavy_nz_off[p.h]);
      const int n = static_cast<int>(heavy_nz_off[p.h + r + 1] - before);
#pragma unroll 4
      for (int j = lane; j < n; j += 32) {
        const V v = a_val[from + j];
        sm.dense[pt.a_u[at + j] * S + r] = v;
        a_bad |= !finite_bits(v);
      }
    }
    a_bad = __syncthreads_or(a_bad);
    for (u32 k = unit.group + warp; k < unit.group + unit.n; k += kPanelWarps) {
      const PanelGroup g = pt.groups[group0 + k];
      const PanelVisit* const visits = pt.visits + entry0 * kPanelVisitsPerEntry + g.first;
      const i64 out = sm.row_out[lane] + pt.group_rows[(group0 + k) * kPanelRows + lane];
      V acc[8][CC];
      u32 rows_of[CH];  // rows that have an entry in the lane's column (of either half)
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < CC; ++j) acc[i][j] = V(0);
#pragma unroll
      for (int c = 0; c < CH; ++c) rows_of[c] = 0u;
      for (int i0 = 0; i0 < static_cast<int>(g.n); i0 += 32) {  // 32 visits' facts, a lane each
        const int n = min(32, static_cast<int>(g.n) - i0);
        u32 l_start = 0, l_u = 0, l_rows = 0, l_lo = 0, l_hi = 0;
        if (lane < n) {
          const PanelVisit v = visits[i0 + lane];
          const GroupPiece piece = pt.pieces[v.piece];
          l_start = piece.start;
          l_lo = static_cast<u32>(piece.mask);
          l_hi = static_cast<u32>(piece.mask >> 32);
          l_u = v.u;
          l_rows = sm.u_mask[v.u];
        }
        V val[D][CH];
        auto request = [&](int d0) {
#pragma unroll
          for (int d = 0; d < D; ++d) {
            const u32 start = __shfl_sync(0xffffffffu, l_start, d0 + d), lo = __shfl_sync(0xffffffffu, l_lo, d0 + d);
            val[d][0] = lo >> lane & 1u ? b_val[start + __popc(lo & lanemask_lt())] : V(0);
            if constexpr (CH > 1) {
              const u32 hi = __shfl_sync(0xffffffffu, l_hi, d0 + d);
              val[d][1] = hi >> lane & 1u ? b_val[start + __popc(lo) + __popc(hi & lanemask_lt())] : V(0);
            }
          }
        };
        request(0);
        for (int d0 = 0; d0 < n; d0 += D) {
          bool bad = a_bad;
#pragma unroll
          for (int d = 0; d < D; ++d)
#pragma unroll
            for (int c = 0; c < CH; ++c) {
              part[d][c * 32 + lane] = val[d][c];
              bad |= !finite_bits(val[d][c]);
            }
          bad = __any_sync(0xffffffffu, bad);
          __syncwarp();
          if (d0 + D < n) request(d0 + D);
#pragma unroll
          for (int d = 0; d < D; ++d) {
            // (past the last visit: a mask and a column of zeros)
            const u32 u = __shfl_sync(0xffffffffu, l_u, d0 + d), rows = __shfl_sync(0xffffffffu, l_rows, d0 + d);
            u32 mask[CH];
            mask[0] = __shfl_sync(0xffffffffu, l_lo, d0 + d);
            if constexpr (CH > 1) mask[1] = __shfl_sync(0xffffffffu, l_hi, d0 + d);
#pragma unroll
            for (int c = 0; c < CH; ++c) rows_of[c] |= mask[c] >> lane & 1u ? rows : 0u;
            V a[8], b[CC];
#pragma unroll
            for (int i = 0; i < 8; i += VEC) *reinterpret_cast<int4*>(a + i) = *reinterpret_cast<const int4*>(&sm.dense[u * S + rg * 8 + i]);
#pragma unroll
            for (int j = 0; j < CC; j += VEC) *reinterpret_cast<int4*>(b + j) = *reinterpret_cast<const int4*>(&part[d][j * 8 + cg * VEC]);
            if (!bad) {
#pragma unroll
              for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < CC; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            } else {
#pragma unroll
              for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < CC; ++j) {
                  const int x = j / VEC * 8 * VEC + cg * VEC + j % VEC;
                  if ((rows >> (rg * 8 + i) & 1u) && (mask[CH > 1 ? j / VEC : 0] >> (x & 31) & 1u)) acc[i][j] = fma(a[i], b[j], acc[i][j]);
                }
            }
          }
          __syncwarp();
        }
      }
      // ---- the group's entries, row by row in column order, four rows at a time through the warp's rows
      const int32_t col0 = static_cast<int32_t>(g.group) * G;
#pragma unroll 1
      for (int quarter = 0; quarter < 4; ++quarter) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (rg == quarter) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < CC; j += VEC)
                *reinterpret_cast<int4*>(&part[i][j * 8 + cg * VEC]) = *reinterpret_cast<const int4*>(&acc[half * 4 + i][j]);
          }
          __syncwarp();
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int row = quarter * 8 + half * 4 + r;
            i64 o = __shfl_sync(0xffffffffu, out, row);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
              const u32 w = __ballot_sync(0xffffffffu, rows_of[c] >> row & 1u);
              if (w >> lane & 1u) {
                const i64 pos = o + __popc(w & lanemask_lt());
                out_col[pos] = col0 + c * 32 + lane;
                out_val[pos] = part[r][c * 32 + lane];
              }
              o += __popc(w);
            }
          }
          __syncwarp();
        }
      }
    }
    if (unit.group == 0) {  // (one block of the panel)
      if (tid < R) task_nnz[row_task_off[p.h + tid] - row_task_off[h0]] = pt.group_rows[(group0 + p.n_groups) * kPanelRows + tid];
      if (tid == 0) atomicAdd(total_rows, static_cast<u64>(R));
    }
  }
}

}  // namespace gm
