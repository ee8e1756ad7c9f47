// K3r — light rows of few products: merged by one thread or sorted by one warp (Algorithm 1 with a sorted accumulator
// instead of a hash table; Section III-E sorts a row after hashing it).
//
//   k3_merge_rows  one thread per row of C: a merge of at most eight (sorted) rows of B.  The heads of the lists live in
//                  registers, every step takes the smallest column and advances all lists that show it.  Nothing is
//                  shared between lanes, so a step costs the instruction stream a few instructions per list for 32
//                  rows at once.
//   k3_sort_rows   one warp per row, up to 1024 products: the products' (column, position) keys are sorted in registers
//                  (see warp_sort_keys), runs of equal columns are added up in the original order.
//
// Both replace the hash accumulator for these sizes.  What bound that one was not memory: a group of lanes cleared a
// table, inserted with compare-and-swap, compacted the table and sorted the entries with a barrier per step, and did the
// first two twice (symbolic, numeric).
//
// Rows either go to the staging area of the light rows at light_off[row], from where k3_copy_rows moves them once
// C.row_ptr is known (one pass over the products, and the entries are written twice), or, when every row of the matrix
// is merged, they are counted first and then written to their place in C: a second merge is cheaper than the copy.
// Without heavy and hashed rows nobody makes C.row_ptr first: k3_place_rows, or the second merge, finds its rows' place in C
// from sums over groups of rows, and writes C.row_ptr too (see RowSums).
#pragma once
#include <type_traits>

#include "gm_common.cuh"
#include "gm_k1_analysis.cuh"
#include "gm_sort.cuh"

namespace gm {

// ------------------------------------------------------------------------------------------------------------------
// merge
// ------------------------------------------------------------------------------------------------------------------
constexpr int kMergeThreads = 128;
constexpr int kMergeStageEntries = 2048;  // entries of C one block collects in shared memory before it writes them out

// kMergePlace: kMergeToC for a block that finds its rows' place in C itself.
enum MergeMode { kMergeCount = 0, kMergeToC = 1, kMergeToStage = 2, kMergePlace = 3 };

// Without heavy rows (and up to kSumRowsMax rows) there is no prefix sum over the rows: whoever counts a row's entries adds them to
// the sum of its group of kSumRows rows, and a block that writes rows to C adds up the groups before its own.  Two launches and
// a pass less (us a call, with the prefix sum / without: 5-point grids of 1024^2 points fp64 250 / 243, of 300^2 86 / 78; ER, 4096 rows of
// 8 73 / 69, 100000 rows of 4 113 / 103, an execute of 30011 rows of 12 fp64 111 / 107 to 112).
// The sums of the next execute are cleared by this one, which the next has waited for.
// Above 256 groups, 64 of them together have a sum of their own, so that a block loads a few values per thread, all at once.  (Fewer
// rows add to few of those, one after the other: ER, 5000 rows of 5 fp64, 39 us an execute with them, 36 without.)
constexpr int kSumRows = 256, kSumGroups = 64;
constexpr i64 kSumDirect = 256;
// Also where C's room waits for the total (see kCRoomBytes; with the prefix sum / without: the 1024^2 grid fp64 258 / 245, of 700^2
// 159 / 158, an execute of ER of 400000 rows of 10 fp32 639 / 633, product of 10^6 rows of 12 2340 / 2348).  Above 2^20 rows it is even or a
// loss: with 2^21 allowed the 1448^2 grid fp32 334 / 340, fp64 399 / 405, ER of 1.5 M rows of 6 2137 / 2126.
constexpr i64 kSumRowsMax = i64{1} << 20;
struct RowSums {
  u32* now;   // nullptr: offsets come from a prefix sum
  u32* next;
  i64 n_groups;  // the sums of groups of groups lie behind those of the groups
};
__device__ __forceinline__ void add_entries(const RowSums& rs, i64 row, u32 n) {
  atomicAdd(&rs.now[row / kSumRows], n);
  if (rs.n_groups > kSumDirect) atomicAdd(&rs.now[rs.n_groups + row / (kSumRows * kSumGroups)], n);
}
// Entries of C before row r0, a multiple of 16 (at least, and of the rows a block has).  All T threads of the block; s_tmp: 33 values.
template <int T>
__device__ __forceinline__ i64 entries_before(const RowSums& rs, const int32_t* __restrict__ row_nnz, i64 r0, i64* s_tmp) {
  static_assert(kSumRowsMax / (kSumRows * kSumGroups) <= T && kSumGroups <= T && kSumDirect <= 2 * T && kSumRows <= 2 * T, "a value of each kind per thread");
  const i64 group = r0 / kSumRows, super = rs.n_groups > kSumDirect ? group / kSumGroups : 0;
  const int t = threadIdx.x;
  const i64 g = super * kSumGroups + t, r = group * kSumRows + t;
  const u32 a = t < super ? rs.now[rs.n_groups + t] : 0u, b = g < group ? rs.now[g] : 0u;
  const u32 b2 = g + T < group ? rs.now[g + T] : 0u;  // (T = 128: up to 256 groups without supers)
  const int c = r < r0 ? row_nnz[r] : 0, d = r + T < r0 ? row_nnz[r + T] : 0;
  const i64 n = static_cast<i64>(a) + b + b2 + c + d;
  i64 total;
  block_exclusive_scan(n, s_tmp, &total);
  return total;
}
__device__ __forceinline__ void clear_next_sums(const RowSums& rs, i64 n_rows) {
  const i64 n = rs.n_groups + (n_rows + kSumRows * kSumGroups - 1) / (kSumRows * kSumGroups);
  for (i64 g = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; g < n; g += static_cast<i64>(gridDim.x) * blockDim.x) rs.next[g] = 0u;
}
// Entries of C in all, for a host that waits for them before it allocates C.  One block of 256 threads.
__global__ void __launch_bounds__(256) k3_total(RowSums rs, i64 n_rows, i64* __restrict__ host_total) {
  static_assert(kSumDirect <= 256 && kSumRowsMax / (kSumRows * kSumGroups) <= 256, "a value per thread");
  __shared__ i64 s_tmp[33];
  const bool direct = rs.n_groups <= kSumDirect;
  const i64 n = direct ? rs.n_groups : (n_rows + kSumRows * kSumGroups - 1) / (kSumRows * kSumGroups);
  i64 total;
  block_exclusive_scan(threadIdx.x < n ? static_cast<i64>(rs.now[(direct ? 0 : rs.n_groups) + threadIdx.x]) : i64{0}, s_tmp, &total);
  if (threadIdx.x == 0) *host_total = total;  // (read after a synchronisation)
}

// One row.  emit(i, column, sum) for the row's i-th entry; returns the number of entries.
template <typename V, int NL, bool NUMERIC, typename Emit>
__device__ __forceinline__ int merge_row(i64 s, i64 e, const int32_t* __restrict__ a_col, const V* __restrict__ a_val,
                                         const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col,
                                         const V* __restrict__ b_val, Emit emit) {
  i64 base[NL];
  int at[NL], len[NL];
  int32_t head[NL];
  V hv[NL], av[NL];  // (a head's value is loaded with its column: one latency per step, not two)
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    base[l] = 0; at[l] = 0; len[l] = 0; av[l] = V(0); hv[l] = V(0);
    if (s + l < e) {
      const int32_t k = a_col[s + l];
      base[l] = b_row_ptr[k];
      len[l] = static_cast<int>(b_row_ptr[k + 1] - base[l]);
      if (NUMERIC) av[l] = a_val[s + l];
    }
  }
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    head[l] = INT_MAX;
    if (len[l] > 0) {
      head[l] = b_col[base[l]];
      if (NUMERIC) hv[l] = b_val[base[l]];
    }
  }
  int n = 0;
  for (;;) {
    int32_t m = head[0];
#pragma unroll
    for (int l = 1; l < NL; ++l) m = min(m, head[l]);
    if (m == INT_MAX) break;  // (columns are below INT_MAX: n_cols <= INT_MAX)
    V sum = V(0);
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      if (head[l] == m) {
        if (NUMERIC) sum += av[l] * hv[l];
        ++at[l];
        head[l] = INT_MAX;
        if (at[l] < len[l]) {
          head[l] = b_col[base[l] + at[l]];
          if (NUMERIC) hv[l] = b_val[base[l] + at[l]];
        }
      }
    }
    emit(n, m, sum);
    ++n;
  }
  return n;
}

// MODE kMergeCount / kMergeToC: rows 0 .. n_rows - 1 in order; kMergeToStage: the rows of a list.
template <typename V, int NL, int MODE>
__global__ void __launch_bounds__(kMergeThreads) k3_merge_rows(
    const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col, const V* __restrict__ a_val,
    const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, const V* __restrict__ b_val,
    const int32_t* __restrict__ rows, i64 n_rows, const i64* __restrict__ light_off, int32_t* __restrict__ row_nnz,
    i64* __restrict__ c_row_ptr, int32_t* __restrict__ out_col, V* __restrict__ out_val, RowSums rs, i64* __restrict__ host_total) {
  const i64 i = static_cast<i64>(blockIdx.x) * kMergeThreads + threadIdx.x;
  const u32 lanes = __ballot_sync(0xffffffffu, i < n_rows);
  if constexpr (MODE == kMergeToC || MODE == kMergePlace) {
    // the block's rows are consecutive, and so are their entries in C: collected in shared memory, written in one run
    // (a thread writing its own entries would touch one sector per lane and store)
    __shared__ int32_t s_col[kMergeStageEntries];
    __shared__ V s_val[kMergeStageEntries];
    const i64 r0 = static_cast<i64>(blockIdx.x) * kMergeThreads;
    const i64 r1 = min(n_rows, r0 + kMergeThreads);
    i64 c0, n_out;
    int at = 0;
    if constexpr (MODE == kMergePlace) {
      __shared__ i64 s_tmp[33];
      __shared__ int s_scan[33];
      int n_all;
      at = block_exclusive_scan(i < n_rows ? row_nnz[i] : 0, s_scan, &n_all);
      c0 = entries_before<kMergeThreads>(rs, row_nnz, r0, s_tmp);
      n_out = n_all;
      if (i < n_rows) c_row_ptr[i] = c0 + at;
      if (i == n_rows - 1) {
        c_row_ptr[n_rows] = c0 + n_out;
        *host_total = c0 + n_out;  // (read after a synchronisation)
      }
      clear_next_sums(rs, n_rows);
    } else {
      c0 = c_row_ptr[r0];
      n_out = c_row_ptr[r1] - c0;
      if (i < n_rows) at = static_cast<int>(c_row_ptr[i] - c0);
    }
    if (n_out <= kMergeStageEntries) {
      if (i < n_rows) {
        merge_row<V, NL, true>(a_row_ptr[i], a_row_ptr[i + 1], a_col, a_val, b_row_ptr, b_col, b_val, [&](int q, int32_t c, V v) {
          s_col[at + q] = c;
          s_val[at + q] = v;
        });
      }
      __syncthreads();
      for (int q = threadIdx.x; q < static_cast<int>(n_out); q += kMergeThreads) {
        out_col[c0 + q] = s_col[q];
        out_val[c0 + q] = s_val[q];
      }
    } else if (i < n_rows) {
      merge_row<V, NL, true>(a_row_ptr[i], a_row_ptr[i + 1], a_col, a_val, b_row_ptr, b_col, b_val, [&](int q, int32_t c, V v) {
        out_col[c0 + at + q] = c;
        out_val[c0 + at + q] = v;
      });
    }
  } else if (i < n_rows) {
    const i64 row = MODE == kMergeToStage ? static_cast<i64>(rows[i]) : i;
    const i64 at = MODE == kMergeToStage ? light_off[row] : 0;
    const int n = merge_row<V, NL, MODE == kMergeToStage>(
        a_row_ptr[row], a_row_ptr[row + 1], a_col, a_val, b_row_ptr, b_col, b_val, [&](int q, int32_t c, V v) {
          if constexpr (MODE == kMergeToStage) {
            out_col[at + q] = c;
            out_val[at + q] = v;
          }
        });
    row_nnz[row] = n;
    if (rs.now) {
      if constexpr (MODE == kMergeCount) {  // a warp's rows are in one group
        const u32 sum = __reduce_add_sync(lanes, static_cast<u32>(n));
        if ((threadIdx.x & 31) == 0) add_entries(rs, row, sum);
      } else {
        add_entries(rs, row, static_cast<u32>(n));
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------------------------
// sort
// ------------------------------------------------------------------------------------------------------------------
// warps per block: what 48 KB of shared memory hold
template <int KMAX> constexpr int kSortWarpsOf = KMAX > 16 ? 2 : 4;
template <int K> constexpr int kSortPosBits = 5 + (K == 1 ? 0 : K == 2 ? 1 : K == 4 ? 2 : K == 8 ? 3 : K == 16 ? 4 : 5);

// Lists of the classes one launch handles, longest rows first.
struct SortLists {
  const int32_t* rows[kSortClasses];
  i64 n[kSortClasses];
};

template <typename V, typename Key, int KMAX>
struct SortSmem {
  i64 base[32];   // per (non-empty) row of B of the current 32 entries of A: its start minus its first product
  V a[32];
  V val[32 * KMAX];
  alignas(16) Key key[32 * KMAX];
};

// The products of A[s..e) into sm.key / sm.val; returns how many.
template <typename V, typename Key, int K, int KMAX>
__device__ __forceinline__ int gather_row(i64 s, i64 e, const int32_t* __restrict__ a_col, const V* __restrict__ a_val,
                                          const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col,
                                          const V* __restrict__ b_val, SortSmem<V, Key, KMAX>& sm) {
  constexpr int kPosBits = kSortPosBits<K>;
  constexpr int U = K >= 4 ? 4 : K;  // windows of 32 products in flight
  const int lane = threadIdx.x & 31;
  int done = 0;
  for (i64 j0 = s; j0 < e; j0 += 32) {
    const i64 j = j0 + lane;
    i64 b0 = 0;
    int len = 0;
    V av = V(0);
    if (j < e) {
      const int32_t k = a_col[j];
      av = a_val[j];
      b0 = b_row_ptr[k];
      len = static_cast<int>(b_row_ptr[k + 1] - b0);
    }
    const u32 some = __ballot_sync(0xffffffffu, len > 0);
    const int inc = warp_inclusive_scan(len);
    const int ex = inc - len;
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    if (len > 0) {
      const int p = __popc(some & lanemask_lt());
      sm.base[p] = b0 - ex;
      sm.a[p] = av;
    }
    __syncwarp();
    int started = 0;  // rows of B that start before the window
    for (int f0 = 0; f0 < total; f0 += 32 * U) {
      int32_t c[U];
      V v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        // which row of B a product belongs to: the rows that start inside the window, as a bit mask over its positions
        const int w = ex - (f0 + u * 32);
        const u32 heads = __reduce_or_sync(0xffffffffu, (len > 0 && w >= 0 && w < 32) ? 1u << w : 0u);
        const int f = f0 + u * 32 + lane;
        if (f < total) {
          const int q = started + __popc(heads & (lanemask_lt() | (1u << lane))) - 1;
          const i64 src = sm.base[q] + f;
          c[u] = b_col[src];
          v[u] = b_val[src] * sm.a[q];
        }
        started += __popc(heads);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int f = f0 + u * 32 + lane;
        if (f < total) {
          sm.key[done + f] = (static_cast<Key>(static_cast<u32>(c[u])) << kPosBits) | static_cast<Key>(done + f);
          sm.val[done + f] = v[u];
        }
      }
    }
    done += total;
    __syncwarp();
  }
  return done;
}

template <typename V, typename Key, int K, int KMAX>
__device__ __forceinline__ void sort_row(i64 row, const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col,
                                         const V* __restrict__ a_val, const i64* __restrict__ b_row_ptr,
                                         const int32_t* __restrict__ b_col, const V* __restrict__ b_val,
                                         const i64* __restrict__ light_off, int32_t* __restrict__ row_nnz,
                                         int32_t* __restrict__ out_col, V* __restrict__ out_val, const RowSums& rs,
                                         SortSmem<V, Key, KMAX>& sm) {
  constexpr int kPosBits = kSortPosBits<K>;
  const int lane = threadIdx.x & 31;
  const i64 at = light_off[row];
  const int n = gather_row<V, Key, K, KMAX>(a_row_ptr[row], a_row_ptr[row + 1], a_col, a_val, b_row_ptr, b_col, b_val, sm);
  int m = 0;
  auto sort = [&](auto width) {
    constexpr int W = decltype(width)::value;
    Key key[W];
#pragma unroll
    for (int r = 0; r < W; ++r) {
      const int q = r * 32 + lane;
      key[r] = q < n ? sm.key[q] : ~Key(0);  // padding sorts to the end
    }
    __syncwarp();
    warp_sort_keys<Key, W>(key, lane);
    m = warp_sum_runs<V, Key, W, kPosBits>(key, n, sm.key, sm.val, 0u, out_col + at, out_val + at);
  };
  if (K == 8 && n <= 160) sort(std::integral_constant<int, 5>{});
  else if (K == 8 && n <= 192) sort(std::integral_constant<int, 6>{});
  else if (K == 4 && n <= 96) sort(std::integral_constant<int, 3>{});
  else sort(std::integral_constant<int, K>{});
  if (lane == 0) {
    row_nnz[row] = m;
    if (rs.now) add_entries(rs, row, static_cast<u32>(m));
  }
  __syncwarp();  // the warp's shared memory is reused by its next row
}

// Warps take rows in list order; SortLists holds the classes K = KMAX, KMAX / 2, ... (n = 0: no such rows).
template <typename V, typename Key, int KMAX>
__global__ void __launch_bounds__(kSortWarpsOf<KMAX> * 32, KMAX > 4 ? 8 : 12) k3_sort_rows(
    const i64* __restrict__ a_row_ptr, const int32_t* __restrict__ a_col, const V* __restrict__ a_val,
    const i64* __restrict__ b_row_ptr, const int32_t* __restrict__ b_col, const V* __restrict__ b_val, SortLists lists,
    const i64* __restrict__ light_off, int32_t* __restrict__ row_nnz, int32_t* __restrict__ out_col, V* __restrict__ out_val,
    RowSums rs) {
  constexpr int kSortWarps = kSortWarpsOf<KMAX>;
  __shared__ SortSmem<V, Key, KMAX> s_sm[kSortWarps];
  SortSmem<V, Key, KMAX>& sm = s_sm[threadIdx.x >> 5];
  const i64 n_warps = static_cast<i64>(gridDim.x) * kSortWarps;
  const i64 w0 = static_cast<i64>(blockIdx.x) * kSortWarps + (threadIdx.x >> 5);
  i64 before = 0;
#define GM_SORT_CLASS(I, K)                                                                                                   \
  if constexpr (K <= KMAX) {                                                                                                  \
    /* the warps go on round-robin from one class to the next */                                                              \
    for (i64 q = ((w0 - before) % n_warps + n_warps) % n_warps; q < lists.n[I]; q += n_warps)                                  \
      sort_row<V, Key, K, KMAX>(lists.rows[I][q], a_row_ptr, a_col, a_val, b_row_ptr, b_col, b_val, light_off, row_nnz, out_col, \
                                out_val, rs, sm);                                                                               \
    before += lists.n[I];                                                                                                     \
  }
  if constexpr (KMAX > 16) {
    GM_SORT_CLASS(0, 32)
  } else if constexpr (KMAX > 4) {
    GM_SORT_CLASS(0, 16)
    GM_SORT_CLASS(1, 8)
  } else {
    GM_SORT_CLASS(0, 4)
    GM_SORT_CLASS(1, 2)
    GM_SORT_CLASS(2, 1)
  }
#undef GM_SORT_CLASS
}

// ------------------------------------------------------------------------------------------------------------------
// staged rows -> C
// ------------------------------------------------------------------------------------------------------------------
// LPR lanes per row of [r0, r1).
template <typename V, int LPR>
__global__ void __launch_bounds__(256) k3_copy_rows(const int32_t* __restrict__ s_col, const V* __restrict__ s_val,
                                                    const i64* __restrict__ light_off, i64 r0, i64 r1,
                                                    const i64* __restrict__ c_row_ptr, int32_t* __restrict__ c_col,
                                                    V* __restrict__ c_val, i64 c_capacity, int* __restrict__ err) {
  const i64 row = r0 + (static_cast<i64>(blockIdx.x) * 256 + threadIdx.x) / LPR;
  const int l = threadIdx.x % LPR;
  if (row >= r1) return;
  const i64 src = light_off[row];
  if (src < 0) return;
  const i64 dst = c_row_ptr[row];
  const int n = static_cast<int>(c_row_ptr[row + 1] - dst);
  if (dst + n > c_capacity) {
    if (l == 0) dev_set_error(err, kDevCapacity);
    return;
  }
#pragma unroll 4
  for (int q = l; q < n; q += LPR) {
    c_col[dst + q] = s_col[src + q];
    c_val[dst + q] = s_val[src + q];
  }
}

template <int LPR> constexpr int kPlaceRows = 256 / LPR * 2;  // rows of a block
// The same for all rows of a product without heavy rows; a block finds the place of its rows itself.
template <typename V, int LPR>
__global__ void __launch_bounds__(256) k3_place_rows(const int32_t* __restrict__ s_col, const V* __restrict__ s_val,
                                                     const i64* __restrict__ light_off, i64 n_rows, const int32_t* __restrict__ row_nnz,
                                                     RowSums rs, i64* __restrict__ c_row_ptr, int32_t* __restrict__ c_col,
                                                     V* __restrict__ c_val, i64 c_capacity, i64* __restrict__ host_total,
                                                     int* __restrict__ err) {
  constexpr int R = kPlaceRows<LPR>;
  static_assert(kSumRows % R == 0 && R <= 256, "a block's rows are in one group");
  __shared__ i64 s_tmp[33];
  __shared__ i64 s_at[R + 1];
  const i64 r0 = static_cast<i64>(blockIdx.x) * R;
  const int n = threadIdx.x < R && r0 + threadIdx.x < n_rows ? row_nnz[r0 + threadIdx.x] : 0;
  const i64 before = entries_before<256>(rs, row_nnz, r0, s_tmp);
  __syncthreads();
  i64 total;
  const i64 at = before + block_exclusive_scan(static_cast<i64>(n), s_tmp, &total);
  if (threadIdx.x < R) {
    s_at[threadIdx.x] = at;
    if (r0 + threadIdx.x < n_rows) c_row_ptr[r0 + threadIdx.x] = at;
    if (r0 + threadIdx.x == n_rows - 1) {
      c_row_ptr[n_rows] = at + n;
      *host_total = at + n;  // (read after a synchronisation)
    }
  }
  if (threadIdx.x == 0) s_at[R] = before + total;
  clear_next_sums(rs, n_rows);
  __syncthreads();
  const int l = threadIdx.x % LPR;
#pragma unroll 1
  for (int i = threadIdx.x / LPR; i < R; i += 256 / LPR) {
    const i64 dst = s_at[i];
    const int m = static_cast<int>(s_at[i + 1] - dst);
    if (m == 0) continue;
    const i64 src = light_off[r0 + i];
    if (dst + m > c_capacity) {
      if (l == 0) dev_set_error(err, kDevCapacity);
      continue;
    }
#pragma unroll 4
    for (int q = l; q < m; q += LPR) {
      c_col[dst + q] = s_col[src + q];
      c_val[dst + q] = s_val[src + q];
    }
  }
}

}  // namespace gm
