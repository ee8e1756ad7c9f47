// C ABI of the library (see include/gmagnus.h): plan = setup phase of Algorithm 3, execute = the
// light and heavy paths, batching of the heavy rows and assembly of C.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "gm_common.cuh"
#include "gm_k1_analysis.cuh"
#include "gm_k3_light.cuh"
#include "gm_k3_rows.cuh"
#include "gm_k4_expand.cuh"
#include "gm_k4_direct.cuh"
#include "gm_k4_stream.cuh"
#include "gm_k4_csc.cuh"
#include "gm_k5_multisplit.cuh"
#include "gm_k6_accumulate.cuh"
#include "gm_k6_panels.cuh"
#include "gm_k6_tasks.cuh"
#include "gm_k7_gather.cuh"
#include "gm_planner.h"
#include "gm_scan.cuh"
#include "gmagnus.h"

namespace gm {

// ------------------------------------------------------------------------------------------------
// errors, allocator
// ------------------------------------------------------------------------------------------------
static thread_local std::string g_last_error;

static int fail(int code, const std::string& msg) {
  g_last_error = msg;
  return code;
}

#define GM_CUDA(expr)                                                                              \
  do {                                                                                             \
    cudaError_t e_ = (expr);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return fail(GM_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_));               \
  } while (0)

#define GM_TRY(expr)                \
  do {                              \
    int rc_ = (expr);               \
    if (rc_ != GM_OK) return rc_;   \
  } while (0)

struct Allocator {
  gm_alloc_fn alloc = nullptr;
  gm_free_fn free = nullptr;
  void* user = nullptr;
};
static Allocator g_alloc;

static void* default_alloc(size_t bytes, cudaStream_t st) {
  static bool pool_ready = false;
  if (!pool_ready) {
    int dev = 0;
    cudaMemPool_t pool;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
      unsigned long long thr = ~0ull;  // keep freed blocks cached: repeated plans reuse them
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    pool_ready = true;
  }
  void* p = nullptr;
  if (cudaMallocAsync(&p, bytes, st) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}

static void* dev_alloc(size_t bytes, cudaStream_t st) {
  if (bytes == 0) bytes = 16;
  if (g_alloc.alloc) {
    void* p = g_alloc.alloc(bytes, st, g_alloc.user);
    // the kernels use 16-byte accesses into what they are given: a hook that hands out less aligned memory is
    // treated like one that has none
    if (p && reinterpret_cast<uintptr_t>(p) % 256 != 0) {
      if (g_alloc.free) g_alloc.free(p, st, g_alloc.user);
      fail(GM_ERR_OOM, "the allocator hook returned a pointer that is not 256-byte aligned");
      return nullptr;
    }
    return p;
  }
  return default_alloc(bytes, st);
}
static void dev_free(void* p, cudaStream_t st) {
  if (!p) return;
  if (g_alloc.free) g_alloc.free(p, st, g_alloc.user);
  else cudaFreeAsync(p, st);
}

struct Buf {
  void* p = nullptr;
  size_t bytes = 0;
};

// What the host needs to know about a device, looked up once (the memory query goes to the kernel driver: 0.2 to 2.6 ms a
// call on a shared host, more than most products take).
struct DeviceFacts {
  bool known = false;
  int num_sms = 0, smem_optin = 0;
  size_t total_mem = 0;
};
constexpr int kMaxDevices = 64;
static std::mutex g_facts_mutex;
static DeviceFacts g_facts[kMaxDevices];

static int device_facts(DeviceFacts* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return fail(GM_ERR_CUDA, "no CUDA device: this library has no CPU path");
  }
  if (dev < 0 || dev >= kMaxDevices) return fail(GM_ERR_INVALID_ARG, "device index out of range");
  std::lock_guard<std::mutex> lock(g_facts_mutex);
  DeviceFacts& f = g_facts[dev];
  if (!f.known) {
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess || n_dev == 0) {
      cudaGetLastError();
      return fail(GM_ERR_CUDA, "no CUDA device: this library has no CPU path");
    }
    size_t free_b = 0;
    GM_CUDA(cudaDeviceGetAttribute(&f.num_sms, cudaDevAttrMultiProcessorCount, dev));
    GM_CUDA(cudaDeviceGetAttribute(&f.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    GM_CUDA(cudaMemGetInfo(&free_b, &f.total_mem));
    f.known = true;
  }
  *out = f;
  return GM_OK;
}

// Streams that the library needs besides the caller's: taken for a call, given back after it, at most kKeptStreams kept per
// device (creating and destroying one per plan cost more than the overlap gained on millisecond products).  Calls that run at
// the same time have different ones: with one for the device, an execute waited for whatever another's stream was busy with.
constexpr size_t kKeptStreams = 8;
static std::vector<cudaStream_t> g_free_streams[kMaxDevices];

static cudaStream_t take_stream() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return nullptr; }
  {
    std::lock_guard<std::mutex> lock(g_facts_mutex);
    if (!g_free_streams[dev].empty()) {
      cudaStream_t st = g_free_streams[dev].back();
      g_free_streams[dev].pop_back();
      return st;
    }
  }
  cudaStream_t st = nullptr;
  if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); return nullptr; }
  return st;
}
static void give_stream(cudaStream_t st) {  // (the caller has waited for it)
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_facts_mutex);
    if (g_free_streams[dev].size() < kKeptStreams) { g_free_streams[dev].push_back(st); return; }
  }
  cudaStreamDestroy(st);
}

struct SideStream {
  cudaStream_t st = nullptr;
  ~SideStream() { if (st) give_stream(st); }
};

// Page-locked host memory that kernels write to and the host reads after a synchronisation: a plan takes one slot and
// gives it back when it is destroyed.  (Copies to ordinary host variables took 12 to 25 us of host time each.)
struct HostSlot {
  int err[4];            // [0] first device-side problem of an execute, [1] malformed input
  u64 totals[kK1Words];  // K1Totals
  i64 c_total;           // nnz(C)
  i64 n_tasks;           // tasks of the heavy rows
  i64 tail[16];          // copy of gm_plan::c_total
  u64 panels[gm::kPanelCounts];  // copy of PanelTables::counts
};
constexpr int kHostSlotBytes = 512;
static_assert(sizeof(HostSlot) <= kHostSlotBytes, "one slot");
static std::mutex g_slot_mutex;
static std::vector<HostSlot*> g_free_slots;

static HostSlot* take_slot() {
  std::lock_guard<std::mutex> lock(g_slot_mutex);
  if (g_free_slots.empty()) {
    constexpr int kSlab = 64;
    void* slab = nullptr;
    if (cudaHostAlloc(&slab, kSlab * kHostSlotBytes, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    for (int i = kSlab - 1; i >= 0; --i)
      g_free_slots.push_back(reinterpret_cast<HostSlot*>(static_cast<char*>(slab) + i * kHostSlotBytes));
  }
  HostSlot* s = g_free_slots.back();
  g_free_slots.pop_back();
  std::memset(s, 0, kHostSlotBytes);
  return s;
}
static void give_slot(HostSlot* s) {
  if (!s) return;
  std::lock_guard<std::mutex> lock(g_slot_mutex);
  g_free_slots.push_back(s);
}

// ------------------------------------------------------------------------------------------------
// plan
// ------------------------------------------------------------------------------------------------
struct PhaseTimes {
  enum Phase { kLightSym, kLightNum, kExpand, kHist, kSplit, kAccSym, kAccNum, kAccSmall, kAccMid, kScan, kCount };
  struct Rec { int phase; cudaEvent_t a, b; };
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> pool;
  size_t used = 0;
  bool enabled = false;
  cudaEvent_t get() {
    if (used == pool.size()) { cudaEvent_t e; cudaEventCreate(&e); pool.push_back(e); }
    return pool[used++];
  }
  void begin(int phase, cudaStream_t st) {
    if (!enabled) return;
    Rec r{phase, get(), get()};
    cudaEventRecord(r.a, st);
    recs.push_back(r);
  }
  void end(cudaStream_t st) {
    if (!enabled) return;
    cudaEventRecord(recs.back().b, st);
  }
  void reset() { recs.clear(); used = 0; }
  void collect(float* out) {
    for (int i = 0; i < kCount; ++i) out[i] = 0.f;
    for (auto& r : recs) { float ms = 0.f; cudaEventElapsedTime(&ms, r.a, r.b); out[r.phase] += ms; }
  }
  ~PhaseTimes() { for (auto e : pool) cudaEventDestroy(e); }
};

}  // namespace gm

// Where gm_spgemm_host wants C: entries are copied to the host batch by batch, while later batches compute.
struct HostSink {
  int32_t* h_col = nullptr;
  void* h_val = nullptr;
  int64_t capacity = 0;          // entries the host buffers hold
  cudaStream_t copy_stream = nullptr;
  int64_t* h_totals = nullptr;   // pinned: entries of C up to the end of each batch
  std::vector<cudaEvent_t> events;
  int64_t copied = 0;            // entries already on their way to the host
};

struct gm_plan {
  gm_csr A{}, B{};
  int sv = 4;
  size_t smem_bytes = 0;
  gm_plan_opts opts{};
  gm_plan_info info{};
  gm_exec_stats stats{};
  int num_sms = 148, smem_optin = 0;
  cudaStream_t plan_stream = nullptr;
  gm::RowRules rules{};
  gm::i64 class_rows[gm::kRowClasses]{};  // light rows per class (see gm_k1_analysis.cuh)
  gm::i64 staged_light = 0;        // products of the light rows that are merged or sorted
  void* light_stage = nullptr;     // the area, if it is an allocation of its own
  bool light_relist = false;       // the area is gone, the rows have to be listed for the hash accumulator first
  int merge_lists = 0;             // most entries of A in a merged row
  bool merge_only = false;         // every row of A is merged or empty
  bool row_sums = false;           // no prefix sum over the rows (see RowSums)
  gm::u32* sums[2]{};              // this execute's and the next one's
  int sums_at = 0;
  bool sums_dirty = false;         // an execute failed on the way
  gm::LightBins bins{};            // hash rows by entry count, for their numeric pass
  int bin_slots[gm::kMaxLightBins]{};
  gm::HostSlot* slot = nullptr;
  bool pending = false;            // kernels of the plan may still run on plan_stream; ev_fork is recorded behind them
  unsigned long long plan_stream_id = 0;  // (the stream may be gone by the time the plan is used)
  std::vector<gm::Batch> batches;
  std::vector<int32_t> x_heavy_host;
  int64_t max_batch_rows = 0;
  int64_t n_seg = 0;
  std::vector<gm::Buf> owned;
  // device arrays
  int64_t* ip = nullptr;           // nA
  int32_t* heavy_flag = nullptr;   // nA
  int32_t* x_heavy = nullptr;      // nH
  int64_t* heavy_base = nullptr;   // nH + 1
  int64_t* seg_off = nullptr;      // n_seg + 1
  int64_t* seg_bstart = nullptr;   // n_seg
  int64_t* seg_j = nullptr;        // n_seg
  int32_t* seg_brow = nullptr;     // n_seg: row of B the segment copies
  uint32_t* child_bound = nullptr; // n_rows(B) x (F0 + 1): where each level-0 child starts inside a row of B
  uint32_t* seg_prefix = nullptr;  // G: (segments of a batch + 1) x F0
  uint32_t* seg_h = nullptr;       // H: segments of a batch x F0 (G minus the child boundary of the segment's row of B)
  uint32_t* seg_tile_sums = nullptr;
  bool direct = false;             // the expansion writes the level-0 children itself
  bool stream = false;             // ... with the rows of B brought in by bulk copies (needs 16-byte aligned B arrays)
  int32_t* seg_hrow = nullptr;     // n_seg: heavy row (position in the heavy-row list) of every segment
  uint32_t* seg_rec = nullptr;     // segment records of a batch for the bulk-copy expansion (run starts + entry of A)
  // outer-product (CSC) order of the expansion, option expand_order = 1: per batch, the segments sorted by row of B
  bool csc = false;
  int32_t* csc_cnt = nullptr;      // n_rows(B) + 1: segments per row of B
  int64_t* csc_ptr = nullptr;      // n_rows(B) + 1: their exclusive scan (the masked CSC's column pointer)
  gm::u64* csc_cursor = nullptr;   // n_rows(B) + 1: scatter cursors
  int32_t* csc_perm = nullptr;     // segments of a batch in CSC order
  int32_t* csc_len = nullptr;      // their product counts
  int64_t* csc_off = nullptr;      // ... and the exclusive scan: the flattened product space in CSC order
  int small_max = 0, mid_max = 0;  // size classes of the final chunks: <= small_max one warp, <= mid_max one small block
  int exit_max = -1;               // chunks of at most this many products leave the multisplit hierarchy early (-1: none)
  unsigned char* exit_tag[2]{};    // per (parent, child) of a level: where the chunk left the hierarchy (ping-pong)
  unsigned char* parent_tag = nullptr;  // per parent of the level that runs: != 0, not split
  std::vector<int64_t> heavy_nz_off_host;
  int64_t* heavy_nz_off = nullptr; // nH + 1
  int32_t* class_list = nullptr;   // classes x nA: light rows per class
  int64_t* light_off = nullptr;    // nA: a row's place in the light staging area, -1: none
  int32_t* light_col = nullptr;    // light staging area: finished rows, at the place of their products
  void* light_val = nullptr;
  int32_t* num_rows = nullptr;     // bins x nA: hash rows by entry count
  int* num_fill = nullptr;         // 8
  int32_t* row_nnz = nullptr;      // nA
  int64_t* scan_tmp = nullptr;
  int64_t* c_total = nullptr;      // [0] running nnz(C) (device carry), [1] heavy entries, [2] products and [3] entries of
                                   // small chunks, [4] products and [5] entries of mid-size chunks, [6] products and
                                   // [7] chunks that left the hierarchy early, [8] products the levels did not move, [9] rows
                                   // in panels
  int* err = nullptr;              // in the host slot: kernels write it through the mapping
  // heavy workspace
  int32_t* stage_col[2]{};
  void* stage_val[2]{};
  gm::u32* counts = nullptr;       // max_batch_rows * chunks_required
  gm::u64* cursor = nullptr;       // same
  int64_t* level_off[2]{};         // max_batch_rows * chunks_required + 1 each (ping-pong)
  gm::u32* chunk_nnz = nullptr;
  int64_t* chunk_nnz_off = nullptr;
  int64_t* chunk_base = nullptr;   // numeric pass: position in C of every chunk's first entry
  int32_t* mid_list = nullptr;     // accumulate kernels: chunks of the mid-size class
  int32_t* big_list = nullptr;     // ... and of the big class (the longest from the front, the others from the back)
  int* acc_counters = nullptr;     // list lengths and tickets (see k6_classify)
  gm::TileMeta* row_meta = nullptr;   // per tile of the expansion kernel: heavy rows it touches (fused histogram)
  gm::TileMeta* tile_meta = nullptr;  // per tile of the expansion / multisplit kernels: groups it touches
  // heavy rows as tasks (see gm_k6_tasks.cuh): no staged products, no levels
  bool use_tasks = false;
  bool finish = false;             // small product: one block does the counting between the kernels (see k_finish_small)
  gm::TaskRules task_rules{};
  int acc_width = 0, acc_threads = 0, acc_blocks = 0;
  gm::u32* piece_bound = nullptr;  // n_rows(B) x (granules + 1)
  gm::u64* longest_row = nullptr;
  gm::u32* part_cols = nullptr;    // granules x (kMaxParts + 1)
  gm::u32* granule_counts = nullptr;
  gm::u32* row_tasks = nullptr;    // nH
  int64_t* row_task_off = nullptr; // nH + 1
  std::vector<int64_t> task_begin; // per batch (and the end): first task
  void* task_mem[2]{};             // the tables of the tasks
  bool task_replan = false;        // they are gone: the tasks have to be listed again
  gm::HeavyTask* tasks = nullptr;
  int64_t* task_off = nullptr;     // place of a task in the staging area
  int32_t* task_list[3]{};         // small, mid, big
  int* task_counters = nullptr;    // 8 per batch
  int* task_tickets = nullptr;     // 4 per batch: big, mid, panels
  bool use_panels = false;         // neighbouring heavy rows with much the same columns are summed together (gm_k6_panels.cuh)
  gm::PanelTables panels{};
  void* panel_mem = nullptr;       // their lists
  std::vector<int64_t> batch_starts;
  gm::PhaseTimes times;
  HostSink* sink = nullptr;        // set by gm_spgemm_host for the duration of one execute
  bool c_is_passing = false;       // C is copied out and freed at once: what it takes more than its entries does not matter
  // light rows run next to the heavy path on a second stream (Algorithm 3 keeps separate queues for them)
  cudaEvent_t ev_fork = nullptr, ev_light = nullptr;
};

namespace gm {

// Blocks of the mid-size class that must fit an SM, with and without staged products.
constexpr int kMidMinBlocks = 7, kMidMinTaskBlocks = 5;

// Lets a kernel take all the dynamic shared memory there is.  (The limit belongs to the kernel and not to a launch: set to what
// one launch needs, it failed the launch of another host thread whose plan has a larger budget.)
template <auto Kern>
static int allow_smem(const gm_plan* p) {
  static std::atomic<int> fixed{-1};  // static shared memory, known once the kernel is loaded
  int n = fixed.load(std::memory_order_relaxed);
  if (n < 0) {
    cudaFuncAttributes a{};
    GM_CUDA(cudaFuncGetAttributes(&a, Kern));
    n = static_cast<int>(a.sharedSizeBytes);
    fixed.store(n, std::memory_order_relaxed);
  }
  GM_CUDA(cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, p->smem_optin - n));
  return GM_OK;
}

template <typename T>
static int plan_alloc(gm_plan* p, T** out, size_t n, cudaStream_t st) {
  Buf b;
  b.bytes = n * sizeof(T);
  b.p = dev_alloc(b.bytes, st);
  if (!b.p) return fail(GM_ERR_OOM, "device allocation of " + std::to_string(b.bytes) + " bytes failed");
  p->owned.push_back(b);
  p->info.workspace_bytes += static_cast<int64_t>(b.bytes);
  *out = static_cast<T*>(b.p);
  return GM_OK;
}

static void plan_free(gm_plan* p, void* q, cudaStream_t st) {
  for (size_t i = 0; q && i < p->owned.size(); ++i) {
    if (p->owned[i].p != q) continue;
    p->info.workspace_bytes -= static_cast<int64_t>(p->owned[i].bytes);
    p->owned.erase(p->owned.begin() + static_cast<std::ptrdiff_t>(i));
    dev_free(q, st);
    return;
  }
}

// Bytes a plan sets aside for the light rows' staging area before it knows their products: an allocation less (a product call of
// ER with 1000 rows takes 76 us, 84 without; with 10000 87.5 and 92), and nothing a device would miss.
constexpr size_t kLightRoom = size_t{4} << 20;
// C is allocated before its size is known, with room for every product, when that takes at most this much: the call then
// does not wait in the middle for nnz(C), and the allocation overlaps the kernels.  Product calls with the wait and without, us:
// ER of 1000 rows 88 / 76, of 10000 95 / 87.5, of 200000 (165 MB of room) 575 / 566; R-MAT scale 12 fp32 (33 MB) 223 / 215.5,
// scale 13 with 15 edges a vertex (90 MB) 336 / 324.  More room would still gain (some 12 us: the 1024^2 grid fp64 245 / 232), but is memory
// that a caller may not have (314 MB of room for that grid's 163 MB), and where C has to move out of it again the call loses: rows of 15
// and 21 neighbouring columns, 60000 and 20000 rows fp64, 100000 fp32, 294 / 312, 226 / 237, 800 / 820, with up to 336 MB more at the peak.
constexpr i64 kCRoomBytes = i64{64} << 20;
// ... and what the caller then holds for nothing is at most this much, or as much again as C itself takes: with more C is
// moved to arrays of its size, which costs some 20 us (block-dense fp32 of 2400 rows, 14 MB of C in 35 MB of room: 346 us moved,
// 328 kept).
constexpr i64 kCSpareBytes = i64{32} << 20;

// Several device arrays in one allocation: the allocator hook of the Python binding costs a few microseconds a call.
struct Arena {
  struct Item { void** slot; size_t offset; };
  std::vector<Item> items;
  size_t bytes = 0;
  void* base = nullptr;
  template <typename T>
  void add(T** slot, size_t n) {
    items.push_back({reinterpret_cast<void**>(slot), bytes});
    bytes += (n * sizeof(T) + 255) & ~size_t{255};
  }
  void place(void* at) {  // (memory that is there already)
    base = at;
    for (const Item& it : items) *it.slot = static_cast<unsigned char*>(at) + it.offset;
  }
  int commit(gm_plan* p, cudaStream_t st) {
    unsigned char* q = nullptr;
    GM_TRY(plan_alloc(p, &q, bytes, st));
    place(q);
    return GM_OK;
  }
};

// First segment of heavy row h (h = 0 .. rows_heavy); the offsets are on the host only when there are several batches.
static i64 seg_begin(const gm_plan* p, i64 h) {
  if (h == 0) return 0;
  if (h == p->info.rows_heavy) return p->n_seg;
  return p->heavy_nz_off_host[static_cast<size_t>(h)];
}

static unsigned grid_for(i64 n, int threads, int num_sms, int per_sm = 16) {
  i64 g = (n + threads - 1) / threads;
  const i64 cap = static_cast<i64>(num_sms) * per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return static_cast<unsigned>(g);
}

// structure_only: the caller reads row_ptr and col_idx alone (values and dtype are not looked at)
static int check_csr_arg(const gm_csr* M, const char* name, bool structure_only = false) {
  if (!M) return fail(GM_ERR_INVALID_ARG, std::string(name) + " is null");
  if (M->n_rows < 0 || M->n_cols < 0 || M->nnz < 0 || M->n_cols > INT32_MAX || M->n_rows > INT32_MAX)
    return fail(GM_ERR_INVALID_ARG, std::string(name) + ": sizes out of range");
  if (!M->row_ptr || (M->nnz > 0 && (!M->col_idx || (!structure_only && !M->vals))))
    return fail(GM_ERR_INVALID_ARG, std::string(name) + ": null array");
  if (!structure_only && M->dtype != GM_F32 && M->dtype != GM_F64)
    return fail(GM_ERR_DTYPE, std::string(name) + ": unknown dtype");
  return GM_OK;
}

__global__ void k_validate_csr(const i64* __restrict__ row_ptr, const int32_t* __restrict__ col, i64 n_rows, i64 n_cols,
                               i64 nnz, int* __restrict__ bad) {
  for (i64 i = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_rows;
       i += static_cast<i64>(gridDim.x) * blockDim.x) {
    const i64 s = row_ptr[i], e = row_ptr[i + 1];
    if ((i == 0 && s != 0) || e < s || e > nnz || (i == n_rows - 1 && e != nnz)) { *bad = 1; continue; }
    for (i64 k = s; k < e; ++k) {
      const int32_t c = col[k];
      if (c < 0 || c >= n_cols || (k > s && col[k - 1] >= c)) { *bad = 1; break; }
    }
  }
}

static i64 row_sum_groups(i64 n_rows) { return (n_rows + kSumRows - 1) / kSumRows; }
static size_t row_sum_words(i64 n_rows) { return (static_cast<size_t>(row_sum_groups(n_rows) * (kSumGroups + 1) / kSumGroups) + 65) & ~size_t{63}; }

// What the row analysis wants zeroed, at the front of an arena.
struct K1Zeroed {
  K1Totals* totals = nullptr;
  HeavyTile* tiles = nullptr;
  i64* ip = nullptr;
  u32* parts = nullptr;
  u32* sums[2]{};  // row_sum_words each, one after the other
  size_t bytes = 0;
  void add_to(Arena& ar, i64 n_rows) {
    ar.add(&totals, 1);
    ar.add(&tiles, static_cast<size_t>((n_rows + kHeavyRows - 1) / kHeavyRows) + 1);
    ar.add(&ip, static_cast<size_t>(n_rows) + 1);
    ar.add(&parts, static_cast<size_t>(n_rows) + 1);
    for (auto& q : sums) ar.add(&q, row_sum_words(n_rows));
    bytes = ar.bytes;
  }
};

// Row analysis: products per row, classes, totals (waits for them).
static int analyse_rows(gm_plan* p, const K1Zeroed& z, cudaStream_t st) {
  const gm_csr& A = p->A;
  K1Totals ht{};
  if (A.n_rows > 0) {
    GM_CUDA(cudaMemsetAsync(z.totals, 0, z.bytes, st));
    const int T = k1_tile_items(A.n_rows, A.nnz, p->num_sms);
    const bool wide = p->B.n_cols > (i64{1} << 24);
    // (blocks that fit the SMs together: 33 KB of shared memory each, 41 with 64-bit prefix sums)
    const unsigned grid = static_cast<unsigned>(std::min<i64>((A.n_rows + A.nnz + T - 1) / T, static_cast<i64>(p->num_sms) * (wide ? 5 : 6)));
    auto kern = T == kK1Small ? (wide ? k1_rows<kK1Small, i64> : k1_rows<kK1Small, u32>)
                              : (wide ? k1_rows<kK1Large, i64> : k1_rows<kK1Large, u32>);
    kern<<<grid, kK1Threads, 0, st>>>(A.row_ptr, A.col_idx, A.n_rows, A.nnz, p->B.row_ptr, p->rules, z.ip, z.parts, p->heavy_flag,
                                      p->row_nnz, p->light_off, p->class_list, A.n_rows, z.tiles, z.totals, p->slot->totals);
    ++p->info.launches;
    GM_CUDA(cudaGetLastError());
    GM_CUDA(cudaStreamSynchronize(st));
    std::memcpy(&ht, p->slot->totals, sizeof(ht));
  }
  gm_plan_info& info = p->info;
  info.products_total = static_cast<int64_t>(ht.products_total);
  info.products_heavy = static_cast<int64_t>(ht.products_heavy);
  info.products_max_row = static_cast<int64_t>(ht.products_max_row);
  info.c_nnz_upper = static_cast<int64_t>(ht.c_nnz_upper);
  info.rows_heavy = static_cast<int64_t>(ht.rows_heavy);
  info.rows_empty = static_cast<int64_t>(ht.rows_empty);
  info.rows_light = A.n_rows - info.rows_heavy - info.rows_empty;
  info.nnz_a_heavy = static_cast<int64_t>(ht.nnz_a_heavy);
  std::memset(info.light_bin_rows, 0, sizeof(info.light_bin_rows));
  for (int c = 0; c < kRowClasses; ++c) {
    p->class_rows[c] = static_cast<i64>(ht.class_rows[c]);
    info.light_bin_rows[std::min(c, 7)] += p->class_rows[c];
  }
  p->staged_light = static_cast<i64>(ht.staged_light);
  p->merge_lists = static_cast<int>(ht.merge_max_lists);
  p->merge_only = p->class_rows[kMergeClass] > 0 && p->class_rows[kMergeClass] + info.rows_empty == A.n_rows;
  return GM_OK;
}

// Lists the light rows for the hash accumulator, which needs no staging area, and gives that area back if there is one: for
// products whose area is refused, larger than asked for, or in the way of C.
static int light_rows_by_hash(gm_plan* p, cudaStream_t st) {
  const i64 nA = p->A.n_rows;
  p->light_relist = true;
  p->row_sums = false;
  plan_free(p, p->light_stage, st);
  p->light_stage = nullptr;
  p->light_col = nullptr;
  p->light_val = nullptr;
  RowRules& r = p->rules;
  r.merge = 0;
  r.sort_max = 0;
  r.n_hash = p->bins.n_bins;
  for (int b = 0; b < p->bins.n_bins; ++b) r.hash_cap[b] = p->bins.cap[b];
  Arena ar;
  K1Zeroed z;  // (its own: a copy of the plan's products per row may be under way)
  z.add_to(ar, nA);
  int32_t* lists = nullptr;
  ar.add(&lists, static_cast<size_t>(kHashClass0 + r.n_hash) * static_cast<size_t>(nA));
  ar.add(&p->num_rows, static_cast<size_t>(p->bins.n_bins) * static_cast<size_t>(nA));
  ar.add(&p->num_fill, 8);
  GM_TRY(ar.commit(p, st));
  p->class_list = lists;
  GM_TRY(analyse_rows(p, z, st));
  p->light_relist = false;
  return GM_OK;
}

constexpr i64 kMinPieceProducts = 5;

// Most bytes a table per row of B (boundaries of children or of granules) may take: 1 GB, or what a staging buffer of the
// default size takes.
static i64 table_room(const gm_plan* p) {
  return std::max<i64>(i64{1} << 30, std::min<i64>(p->info.products_heavy, i64{1} << 29) * (4 + p->sv));
}

// Sizes of the heavy rows' tasks; false: they do not fit (then the rows go through the staged products).
static bool plan_task_rules(gm_plan* p) {
  const gm_params& prm = p->info.params;
  const gm_plan_opts& o = p->opts;
  if (p->B.nnz >= (i64{1} << 32) || p->B.n_rows == 0) return false;  // piece boundaries are 32-bit positions in B's arrays
  // kBigBlocks accumulators per SM unless another number was asked for
  const int ctas = o.acc_ctas_per_sm == 0 ? kBigBlocks : o.acc_ctas_per_sm;
  const int bt = o.acc_ctas_per_sm == 0 ? kBigThreads : 1024 / ctas;
  const size_t budget = p->smem_bytes / static_cast<size_t>(ctas) - 1024;
  i64 w = prm.chunk_width;
  auto smem = [&](i64 width) { return p->sv == 4 ? big_task_smem_bytes<float>(static_cast<int>(width), bt) : big_task_smem_bytes<double>(static_cast<int>(width), bt); };
  while (w > 32 && smem(w) > budget) w /= 2;
  if (smem(w) > budget) return false;
  const i64 granules = (prm.chunk_width / w) * prm.chunks_required;
  if (granules > 512) return false;
  if ((p->B.n_rows * (granules + 1) + (granules > 1 ? p->info.rows_heavy * granules : 0)) * 4 > table_room(p)) return false;
  p->acc_width = static_cast<int>(w);
  p->acc_threads = bt;
  p->acc_blocks = ctas;
  TaskRules& r = p->task_rules;
  r.granules = static_cast<int>(granules);
  r.log2_g = ilog2_floor(static_cast<uint64_t>(w));
  // Sorted by one warp up to 256 products (a chunk of staged products only up to 128: it is read once, where a mid-size task
  // generates its products twice).  R-MAT scale 19 fp32, 128 / 256 / 512: sorts
  // 0.77 / 2.08 / 5.48 ms, mid-size tasks 23.0 / 20.7 / 18.1.
  r.small_max = o.small_chunk_max ? p->small_max : 256;
  r.small_width = 1u << 22;  // a sort key packs the column inside the task with a position of at most nine bits
  const i64 span = static_cast<i64>(pow2_ceil(static_cast<uint64_t>(std::max<i64>(p->B.n_cols, 32))));
  r.mid_width = static_cast<u32>(std::max<i64>(w, std::min<i64>(32768, span)));
  // Hand-over to the dense accumulator: its flush goes with the columns of a granule, the two passes of the mid-size block with the
  // products.  A quarter of the columns (R-MAT scale 19 fp32, 1024 / 2048 / 4096 products: 77 / 67 / 65 ms); an eighth for
  // products that leave most of the device idle, where one block's time counts (scale 10 fp32: 130 us against 149 with all
  // of the columns, scale 12 181 against 195).
  const int mid_default = static_cast<int>(std::max<i64>(256, std::min<i64>(p->sv == 4 ? 4096 : 2048, w / (p->info.products_heavy < (i64{1} << 24) ? 8 : 4))));
  int mid = o.mid_chunk_max < 0 ? 0 : (o.mid_chunk_max ? o.mid_chunk_max : mid_default);
  const size_t fixed = (p->sv == 4 ? sizeof(Pieces<float, kMidThreads * kMidPerThread>) : sizeof(Pieces<double, kMidThreads * kMidPerThread>)) + 2048;
  while (mid > r.small_max && mid_task_smem_bytes(static_cast<int>(r.mid_width), p->sv, mid) + fixed > p->smem_bytes / kMidMinTaskBlocks) mid /= 2;
  r.mid_max = std::max(mid, r.small_max);
  // A hub row's granule is cut when it would keep a block busy for longer than an eighth of its even share of the whole (but
  // not below 8192 products, where the pieces of the sub-ranges get short: R-MAT scale 12 took 312 us with a floor of 32768,
  // 295 with 8192; and only with more products than columns, which is what the sub-ranges' places in the staging area take).
  r.split_above = static_cast<u32>(std::min<i64>(1u << 30, std::max<i64>(std::max<i64>(1 << 13, w), p->info.products_heavy / (static_cast<i64>(p->num_sms) * ctas * 8))));
  r.max_parts = kMaxParts;
  return true;
}

// Panels are looked for where heavy rows have many entries (R-MAT graphs have 25 to 40, and hardly two rows alike; with 8 instead of 48
// R-MAT scale 17 fp64 took 3880 us instead of 3857, ER of 100000 rows of 30 1962 instead of 1927) and where there are products enough to pay
// for the lists.  Block-dense products, us a call, tasks / panels: 2.8 M products fp64 150 / 195, 23 M fp32
// 292 / 319, 43 M fp32 336 / 342, 166 M fp64 (kept plan) 895 / 510, 1.3 G fp64 5690 / 1630, 2.7 G fp32 8560 / 2440.
constexpr i64 kPanelMinEntries = 48, kPanelMinHeavy = i64{1} << 26;
// They are built where what they are expected to save, in products, pays for them (some 50 us and 20 ps an entry of A).
constexpr i64 kPanelMinGain = i64{1} << 25, kPanelGainPerEntry = 16;
constexpr size_t kPanelMemoryShare = 32;  // the lists take at most this part of the device's memory
static int panel_max_u(const gm_plan* p) { return p->sv == 4 ? kPanelColumns<float> : kPanelColumns<double>; }
static i64 panel_groups(const gm_plan* p) { return ((p->B.n_cols - 1) >> panel_group_bits(p->sv)) + 1; }
// Groups of a unit: two for every warp where the panels keep the device busy all the same.  (Block-dense fp32, us with one / two, block rows
// of 40: 3300 heavy rows 358 / 358, 7300 551 / 546, 11200 742 / 712, 16800 917 / 872; fp64 7300 648 / 630, 14000 918 / 868.)
static int panel_unit_groups(i64 n_heavy) { return n_heavy >= kPanelRows * 256 ? 2 * kPanelWarps : kPanelWarps; }
static bool plan_panel_rules(const gm_plan* p) {
  const size_t smem = p->sv == 4 ? sizeof(PanelSmem<float>) : sizeof(PanelSmem<double>);
  return p->info.products_heavy >= kPanelMinHeavy && p->n_seg >= kPanelMinEntries * p->info.rows_heavy && p->B.n_rows <= kPanelMaxRowsB &&
         panel_groups(p) <= kPanelMaxGroups && std::max(smem, panel_build_smem(p->B.n_rows, panel_groups(p))) + 1024 <= p->smem_bytes;
}

// No panels after all: the lists are given back (nothing that is queued uses them), the rows are tasks like the others.
static void drop_panels(gm_plan* p, cudaStream_t st) {
  p->use_panels = false;
  plan_free(p, p->panel_mem, st);
  p->panel_mem = nullptr;
}

// The lists of the panels, sized by what was found (in the host slot).  Nothing is allocated where that does not pay: for ER of 20000
// rows of 60 fp32, no two rows alike, lists for all heavy rows took 38 us of 915 and 62 MB.
static int build_panels(gm_plan* p, cudaStream_t st) {
  const gm_csr& A = p->A;
  const gm_csr& B = p->B;
  const i64 nH = p->info.rows_heavy;
  PanelTables& pt = p->panels;
  const u64* const found = p->slot->panels;
  const size_t entries = static_cast<size_t>(found[kPanelEntries]), groups = entries / kPanelEntriesPerGroup + 1;
  u32* piece_count = nullptr;
  i64* piece_tmp = nullptr;
  Arena ar, scratch;
  ar.add(&pt.a_u, entries);
  ar.add(&pt.u_mask, entries);
  ar.add(&pt.groups, groups);
  ar.add(&pt.group_rows, groups * kPanelRows);
  ar.add(&pt.units, groups);
  ar.add(&pt.piece_ptr, static_cast<size_t>(B.n_rows) + 1);
  pt.max_pieces = B.nnz / kPanelEntriesPerPiece + 1;
  ar.add(&pt.pieces, static_cast<size_t>(pt.max_pieces));
  // (what only the prefix sum over the pieces needs lies where the visits will be)
  scratch.add(&piece_count, static_cast<size_t>(B.n_rows));
  scratch.add(&piece_tmp, static_cast<size_t>(scan_tmp_elems(B.n_rows)));
  ar.add(&pt.visits, std::max(entries * kPanelVisitsPerEntry, scratch.bytes / sizeof(PanelVisit) + 1));
  DeviceFacts facts;
  GM_TRY(device_facts(&facts));
  if (static_cast<i64>(found[kPanelGain]) < kPanelMinGain + kPanelGainPerEntry * static_cast<i64>(entries) || ar.bytes > facts.total_mem / kPanelMemoryShare || ar.commit(p, st) != GM_OK) {
    p->use_panels = false;  // they do not pay, or there is no room
    return GM_OK;
  }
  p->panel_mem = ar.base;
  scratch.place(pt.visits);
  const int group_bits = panel_group_bits(p->sv), n_groups = static_cast<int>(panel_groups(p));
  const unsigned row_grid = grid_for(B.n_rows, 8, p->num_sms, 16);
  k_piece_count<<<row_grid, 256, 0, st>>>(B.row_ptr, B.col_idx, B.n_rows, group_bits, piece_count);
  p->info.launches += 3 + exclusive_scan<u32, i64>(piece_count, pt.piece_ptr, B.n_rows, piece_tmp, nullptr, nullptr, nullptr, st);
  k_piece_fill<<<row_grid, 256, 0, st>>>(B.row_ptr, B.col_idx, B.n_rows, group_bits, pt);
  GM_TRY(allow_smem<k_panel_build>(p));
  k_panel_build<<<static_cast<unsigned>(std::min<i64>(static_cast<i64>(found[kPanelsFound]), static_cast<i64>(p->num_sms) * 3)), kPanelBuildThreads,
                  panel_build_smem(B.n_rows, n_groups), st>>>(pt, p->x_heavy, p->heavy_base, p->heavy_nz_off, A.row_ptr, A.col_idx, B.n_rows,
                                                              n_groups, panel_max_u(p), panel_unit_groups(nH));
  return GM_OK;
}

// Tasks of the heavy rows: piece boundaries of B, products per row and granule, ranges, lists.
static int plan_tasks(gm_plan* p, cudaStream_t st) {
  const gm_csr& A = p->A;
  const gm_csr& B = p->B;
  const TaskRules& r = p->task_rules;
  const i64 nH = p->info.rows_heavy;
  const size_t n_batches = p->batches.size();
  u32* n_long = nullptr;
  int32_t* long_rows = nullptr;
  i64* tmp = nullptr;
  unsigned char* similar = nullptr;
  i64* starts = nullptr;
  PanelTables& pt = p->panels;
  // Small products: the tables take their upper bound (a granule of n products gives fewer than 2 n / split_above
  // sub-ranges), so that nothing waits for the number of tasks.
  const i64 bound = nH * r.granules + 2 * (p->info.products_heavy / r.split_above) + 64;
  p->finish = n_batches == 1 && bound <= kFinishMax && A.n_rows <= kFinishMax;
  auto add_tables = [&](Arena& ar, i64 n_tasks, i64 max_tasks) {
    const size_t n = static_cast<size_t>(n_tasks), m = static_cast<size_t>(max_tasks);
    ar.add(&p->tasks, n);
    ar.add(&p->task_off, n + 1);
    for (auto& l : p->task_list) ar.add(&l, n);
    ar.add(&p->chunk_nnz, m + 1);
    ar.add(&p->chunk_nnz_off, m + 1);
    ar.add(&p->chunk_base, m + 1);
    ar.add(&p->tile_meta, static_cast<size_t>(p->info.stage_elems) / kGatherTile + 2);
    ar.add(&p->scan_tmp, static_cast<size_t>(scan_tmp_elems(std::max<i64>(max_tasks, A.n_rows))));
  };
  {
    Arena ar;
    ar.add(&p->longest_row, 1);
    ar.add(&n_long, 1);
    ar.add(&p->task_counters, 8 * n_batches);
    if (p->use_panels) {
      ar.add(&pt.counts, kPanelCounts);
      ar.add(&starts, n_batches);
    }
    const size_t zeroed = ar.bytes;
    if (p->use_panels) {
      ar.add(&pt.list, static_cast<size_t>(nH) / kPanelMinRows + 1);
      ar.add(&pt.of_row, static_cast<size_t>(nH));
      ar.add(&similar, static_cast<size_t>(nH));
    }
    ar.add(&p->c_total, 16);  // (next to the tickets: one clear for both, see execute_t)
    ar.add(&p->task_tickets, 4 * n_batches);
    ar.add(&p->piece_bound, static_cast<size_t>(B.n_rows) * static_cast<size_t>(r.granules + 1));
    ar.add(&p->part_cols, static_cast<size_t>(r.granules) * (kMaxParts + 1));
    ar.add(&p->row_tasks, static_cast<size_t>(nH));
    ar.add(&p->row_task_off, static_cast<size_t>(nH) + 1);
    ar.add(&tmp, static_cast<size_t>(scan_tmp_elems(nH)));
    if (r.granules > 1) {
      ar.add(&p->granule_counts, static_cast<size_t>(nH) * static_cast<size_t>(r.granules));
      ar.add(&long_rows, static_cast<size_t>(nH));
    }
    if (p->finish) add_tables(ar, bound, bound);
    GM_TRY(ar.commit(p, st));
    p->task_mem[0] = ar.base;
    GM_CUDA(cudaMemsetAsync(p->longest_row, 0, zeroed, st));
  }
  if (p->use_panels) {
    if (n_batches > 1) {
      p->batch_starts.clear();
      for (const Batch& b : p->batches) p->batch_starts.push_back(b.h0);
      GM_CUDA(cudaMemcpyAsync(starts, p->batch_starts.data(), n_batches * sizeof(i64), cudaMemcpyHostToDevice, st));
    }
    k_panel_similar<<<static_cast<unsigned>((nH + 7) / 8), 256, 0, st>>>(p->x_heavy, nH, A.row_ptr, A.col_idx, B.row_ptr, B.col_idx,
                                                                       panel_group_bits(p->sv), pt.counts, similar);
    k_panel_cut<<<static_cast<unsigned>((nH + 1023) / 1024), 1024, 0, st>>>(similar, nH, starts, static_cast<int>(n_batches), p->heavy_base,
                                                                          p->heavy_nz_off, static_cast<int>(panel_groups(p)), panel_unit_groups(nH),
                                                                          p->sv == 4 ? kPanelCost<float> : kPanelCost<double>, pt, p->slot->panels);
    p->info.launches += 2;
    if (!p->ev_light) GM_CUDA(cudaEventCreateWithFlags(&p->ev_light, cudaEventDisableTiming));
    GM_CUDA(cudaEventRecord(p->ev_light, st));
  }
  k_piece_bounds<<<grid_for(B.n_rows * (r.granules + 1), 256, p->num_sms, 32), 256, 0, st>>>(B.row_ptr, B.col_idx, B.n_rows, r.granules,
                                                                                           r.log2_g, p->piece_bound, p->longest_row);
  k_granule_parts<<<static_cast<unsigned>(r.granules), 32, 0, st>>>(B.col_idx, p->piece_bound, p->longest_row, r.granules, r.log2_g,
                                                                  p->part_cols);
  p->info.launches += 2;
  if (p->use_panels) {
    GM_CUDA(cudaEventSynchronize(p->ev_light));  // (while the two kernels before this run)
    GM_TRY(build_panels(p, st));
  }
  const unsigned char* in_panel = p->use_panels ? p->panels.of_row : nullptr;
  if (r.granules > 1) {
    k_granule_counts<<<grid_for(nH, 8, p->num_sms, 8), 256, 0, st>>>(p->x_heavy, nH, A.row_ptr, A.col_idx, p->piece_bound, r.granules,
                                                                   p->granule_counts, long_rows, n_long, in_panel);
    k_granule_counts_long<<<static_cast<unsigned>(p->num_sms * kCountRuns), 256, 0, st>>>(p->x_heavy, A.row_ptr, A.col_idx, p->piece_bound, r.granules,
                                                                               p->granule_counts, long_rows, n_long);
    p->info.launches += 2;
  }
  p->task_begin.assign(n_batches + 1, 0);
  if (p->finish) {
    p->task_begin[1] = bound;
    const TaskTables tt{p->tasks, p->task_off, {p->task_list[0], p->task_list[1], p->task_list[2]}, p->task_counters, 0, bound};
    k_plan_small<<<1, kFinishThreads, 0, st>>>(p->granule_counts, p->heavy_base, nH, r, p->row_tasks, p->row_task_off, p->x_heavy, A.row_ptr,
                                              p->part_cols, tt, in_panel);
    ++p->info.launches;
    GM_CUDA(cudaGetLastError());
    return GM_OK;
  }
  k_task_count<<<static_cast<unsigned>((nH + 127) / 128), 128, 0, st>>>(p->granule_counts, p->heavy_base, nH, r, p->row_tasks, in_panel,
                                                                       p->use_panels ? pt.counts : nullptr, p->slot->panels);
  p->info.launches += 1 + exclusive_scan<u32, i64>(p->row_tasks, p->row_task_off, nH, tmp, nullptr, nullptr, nullptr, st,
                                                  reinterpret_cast<i64*>(&p->slot->n_tasks));
  for (size_t i = 1; i < n_batches; ++i)
    GM_CUDA(cudaMemcpyAsync(&p->task_begin[i], p->row_task_off + p->batches[i].h0, sizeof(i64), cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  p->task_begin[n_batches] = p->slot->n_tasks;
  if (p->use_panels && p->slot->panels[kPanelUnits] == 0) {  // none pays (a small product finds that out in its first execute)
    drop_panels(p, st);
    in_panel = nullptr;
  }
  i64 max_tasks = 0;
  for (size_t i = 0; i < n_batches; ++i) max_tasks = std::max(max_tasks, p->task_begin[i + 1] - p->task_begin[i]);
  {
    Arena ar;
    add_tables(ar, p->slot->n_tasks, max_tasks);
    GM_TRY(ar.commit(p, st));
    p->task_mem[1] = ar.base;
  }
  for (size_t i = 0; i < n_batches; ++i) {
    const Batch& b = p->batches[i];
    const TaskTables tt{p->tasks, p->task_off, {p->task_list[0], p->task_list[1], p->task_list[2]}, p->task_counters + 8 * i,
                        p->task_begin[i], p->task_begin[i + 1]};
    k_task_emit<<<static_cast<unsigned>((b.h1 - b.h0 + 127) / 128), 128, 0, st>>>(p->granule_counts, p->heavy_base, b.h0, b.h1, b.elem0, r,
                                                                                p->row_task_off, p->x_heavy, A.row_ptr, p->part_cols, tt, in_panel);
    ++p->info.launches;
  }
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// Lists the heavy rows' tasks again, without panels, whose lists are given back: for products whose C is refused beside them.
static int tasks_without_panels(gm_plan* p, cudaStream_t st) {
  p->task_replan = true;
  drop_panels(p, st);
  for (auto& q : p->task_mem) {
    plan_free(p, q, st);
    q = nullptr;
  }
  GM_TRY(plan_tasks(p, st));
  p->task_replan = false;
  return GM_OK;
}

static int build_plan(gm_plan* p, cudaStream_t st) {
  const gm_csr& A = p->A;
  const gm_csr& B = p->B;
  const i64 nA = A.n_rows;
  gm_plan_info& info = p->info;
  info.n_rows = nA;
  info.n_cols_c = B.n_cols;

  DeviceFacts facts;
  GM_TRY(device_facts(&facts));
  p->num_sms = facts.num_sms;
  p->smem_optin = facts.smem_optin;
  if (p->smem_bytes > static_cast<size_t>(facts.smem_optin))
    return fail(GM_ERR_UNSUPPORTED_SMEM, "smem_bytes exceeds the device's opt-in shared memory per block");
  {
    const int rc = planner_params(B.n_cols, A.dtype, p->smem_bytes, &p->opts, &info.params);
    if (rc != GM_OK) return fail(rc, "planner rejected the parameters");
  }
  const gm_params& prm = info.params;
  {
    // size classes of the final chunks (Section III-E bins chunks by size)
    const gm_plan_opts& o = p->opts;
    if (o.small_chunk_max < -1 || o.small_chunk_max > kAccSmallChunk || o.mid_chunk_max < -1 || o.mid_chunk_max > (1 << 15))
      return fail(GM_ERR_INVALID_ARG, "small_chunk_max / mid_chunk_max out of range");
    p->small_max = o.small_chunk_max < 0 ? 0 : (o.small_chunk_max ? o.small_chunk_max : kAccSmallDefault);
    int mid = o.mid_chunk_max < 0 ? 0 : (o.mid_chunk_max ? o.mid_chunk_max : (p->sv == 4 ? 4096 : 2048));
    // several mid-chunk blocks must fit an SM next to each other for the class to pay
    while (mid > p->small_max && mid_smem_bytes(prm.chunk_width, p->sv, mid) + 1024 > p->smem_bytes / kMidMinBlocks) mid /= 2;
    if (prm.chunk_width > 65536) mid = 0;  // the kernel keeps a chunk's columns as 16-bit offsets
    p->mid_max = std::max(mid, p->small_max);
    if (o.early_exit < -1 || o.early_exit > kAccSmallChunk) return fail(GM_ERR_INVALID_ARG, "early_exit out of range");
    // early exit needs the one-warp sort (the only accumulate kernel that takes a chunk wider than W) and a level
    // after the first
    p->exit_max = (o.early_exit < 0 || p->small_max <= 0 || prm.n_levels < 2) ? -1
                  : std::min(o.early_exit ? o.early_exit : p->small_max, p->small_max);
  }

  p->slot = take_slot();
  if (!p->slot) return fail(GM_ERR_OOM, "page-locked host memory for the plan's counters could not be had");
  p->err = p->slot->err;
  if (p->opts.validate_inputs) {
    for (const gm_csr* M : {&A, &B}) {
      if (M->n_rows == 0) continue;
      k_validate_csr<<<grid_for(M->n_rows, 256, p->num_sms), 256, 0, st>>>(M->row_ptr, M->col_idx, M->n_rows,
                                                                          M->n_cols, M->nnz, p->err + 1);
    }
    info.launches += 2;
    GM_CUDA(cudaStreamSynchronize(st));
    if (p->slot->err[1]) return fail(GM_ERR_BAD_CSR, "row_ptr not monotone / columns out of range or not strictly ascending");
  }

  // ---- K1: products per row, classes, totals
  {
    // light rows: merged by a thread (when there are enough rows to fill the device with one thread each), sorted by a
    // warp, or (above kSortMaxProducts: only with a tau that large) hashed
    RowRules& r = p->rules;
    r.tau = prm.tau;
    r.c_cols = B.n_cols;
    r.merge = nA >= kMergeMinRows ? 1 : 0;
    r.sort_max = kSortMaxProducts;
    r.n_hash = 0;
    const int top_cap = static_cast<int>(pow2_ceil(static_cast<uint64_t>(std::max<i64>(prm.tau, 16))));
    for (int c : {1024, 4096, 16384, 65536})
      if (c < top_cap) r.hash_cap[r.n_hash++] = c;
    r.hash_cap[r.n_hash++] = std::max(top_cap, 1024);
    int nb = 0;
    for (int c : {16, 64, 256, 1024, 4096, 16384, 65536})
      if (c < top_cap && nb < kMaxLightBins - 1) { p->bins.cap[nb] = c; p->bin_slots[nb] = 2 * c; ++nb; }
    p->bins.cap[nb] = top_cap;
    p->bin_slots[nb] = prm.light_slots;
    p->bins.n_bins = nb + 1;
  }
  unsigned char* light_room = nullptr;
  K1Zeroed z;
  {
    Arena ar;
    const size_t n1 = static_cast<size_t>(nA) + 1;
    z.add_to(ar, nA);
    ar.add(&p->c_total, 16);
    ar.add(&p->heavy_flag, n1);
    ar.add(&p->row_nnz, n1);
    ar.add(&p->light_off, n1);
    ar.add(&p->class_list, static_cast<size_t>(kHashClass0 + p->rules.n_hash) * n1);
    ar.add(&p->scan_tmp, static_cast<size_t>(scan_tmp_elems(std::max<i64>(nA, 1))));
    ar.add(&light_room, kLightRoom);  // the light rows' staging area, if it turns out to fit: an allocation less
    GM_TRY(ar.commit(p, st));
  }
  p->ip = z.ip;
  GM_TRY(analyse_rows(p, z, st));  // ---- first host sync: totals
  const i64 nH = info.rows_heavy;
  p->n_seg = info.nnz_a_heavy;
  for (int i = 0; i < 2; ++i) p->sums[i] = z.sums[i];

  // ---- light rows: staging area (not when all rows are merged), bins of the hash rows
  bool hash_all = false;
  if (p->staged_light > 0 && !p->merge_only) {
    // at most what a staging buffer of the heavy rows may hold (see below): the area takes room for every product, where C
    // may have one entry for many, and the hash accumulator takes none
    const i64 most = p->opts.stage_elems > 0 ? p->opts.stage_elems : std::max<i64>(i64{1} << 29, static_cast<i64>(facts.total_mem / 5) / (4 + p->sv));
    const size_t n_staged = static_cast<size_t>(p->staged_light) + 64, bytes = n_staged * static_cast<size_t>(4 + p->sv);
    unsigned char* area = light_room;
    if (p->staged_light > most) hash_all = true;
    else if (bytes > kLightRoom) hash_all = plan_alloc(p, &area, bytes, st) != GM_OK;
    if (!hash_all) {
      p->light_stage = area == light_room ? nullptr : area;
      p->light_val = area;
      p->light_col = reinterpret_cast<int32_t*>(area + n_staged * static_cast<size_t>(p->sv));
    }
  }
  if (hash_all) {
    GM_TRY(light_rows_by_hash(p, st));
  } else {
    Arena ar;
    bool hash_rows = false;
    for (int c = kHashClass0; c < kRowClasses; ++c) hash_rows |= p->class_rows[c] > 0;
    if (hash_rows) {
      ar.add(&p->num_rows, static_cast<size_t>(p->bins.n_bins) * static_cast<size_t>(nA));
      ar.add(&p->num_fill, 8);
      GM_TRY(ar.commit(p, st));
    }
    p->row_sums = nH == 0 && !hash_rows && info.rows_empty < nA && nA <= kSumRowsMax;
  }

  // ---- heavy rows
  if (nH > 0) {
    {
      Arena ar;
      ar.add(&p->x_heavy, static_cast<size_t>(nH));
      ar.add(&p->heavy_base, static_cast<size_t>(nH) + 1);
      ar.add(&p->heavy_nz_off, static_cast<size_t>(nH) + 1);
      GM_TRY(ar.commit(p, st));
    }
    k1_heavy_lists<<<static_cast<unsigned>((nA + kHeavyRows - 1) / kHeavyRows), kHeavyThreads, 0, st>>>(
        p->ip, p->heavy_flag, A.row_ptr, nA, z.tiles, p->x_heavy, p->heavy_base, p->heavy_nz_off);
    ++info.launches;

    // The expansion writes the first level's children itself (see gm_k4_direct.cuh) unless asked to run that
    // level as separate histogram and multisplit passes.
    // That takes a row of F0 run starts per segment, which pays when segments are long compared with the
    // fan-out (R-MAT products: ~1000 products per segment) and not when they are short (a clipped-Zipf pair
    // with F0 = 256 and ~60 products per segment measured 3x slower that way).
    const bool long_segments = prm.n_levels > 0 &&
                               info.products_heavy >= 2 * static_cast<i64>(prm.fanout[0]) * std::max<i64>(info.nnz_a_heavy, 1);
    // ... and a table of F0 + 1 boundaries per row of B, which must stay small
    const i64 bound_bytes = prm.n_levels > 0 ? B.n_rows * static_cast<i64>(prm.fanout[0] + 1) * 4 : 0;
    const bool bounds_fit = bound_bytes <= table_room(p);
    p->csc = p->opts.expand_order == 1;
    p->direct = prm.n_levels > 0 && prm.fanout[0] <= 256 && !p->csc &&
                (p->opts.level0_multisplit == 2 || (p->opts.level0_multisplit == 0 && long_segments && bounds_fit));
    {
      const size_t warp_smem = stream_warp_smem_bytes(prm.n_levels > 0 ? prm.fanout[0] : 2, p->sv);
      p->stream = p->direct && p->opts.expand_staging == 1 && reinterpret_cast<uintptr_t>(B.col_idx) % 16 == 0 &&
                  reinterpret_cast<uintptr_t>(B.vals) % 16 == 0 && p->smem_bytes >= kStreamWarps * warp_smem + 1024;
    }
    // Products are summed where they are generated, unless a first level is asked for or the pieces of B's rows get too short: a task looks every row of B up
    // in the boundary table, so that costs per (segment, granule) and not per product.  Products per (segment, granule) and time
    // per call, tasks against staged products: R-MAT scale 18 fp64 with 4 edges a vertex about 9, 4.2 against 5.4 ms; R-MAT scale 20
    // fp32 20, 188 against 198 ms; R-MAT scale 21 fp64 3.7, 291 against 278 ms.  With rows of equal length (ER) 1.9 / 2.5: 3.25
    // against 3.13 ms / 10.4 against 9.95; R-MAT scale 19 fp64 with 4 / 8 edges a vertex 5.1 / 9.0: 10.73 against 10.78 / 30.7 against
    // 33.8.  Up to eight granules it is the pieces of a row that count little: ER of 65536 and 131072 columns, 1.0: 1.90 against 2.05 ms,
    // 1.9: 1.51 against 1.87, 3.75: 1.46 against 1.65 and 2.47 against 2.74, and 7.5 with four granules 1.25 against 1.20.
    p->use_tasks = p->opts.level0_multisplit == 0 && !p->csc && !p->stream && (prm.n_levels == 0 || (prm.n_levels == 1 && p->direct)) && plan_task_rules(p) &&
                   (p->task_rules.granules <= 8 || info.products_heavy >= kMinPieceProducts * p->n_seg * p->task_rules.granules);
    info.heavy_tasks = p->use_tasks ? 1 : 0;
    info.task_ctas_per_sm = p->use_tasks ? p->acc_blocks : 0;
    info.level0_direct = p->direct && !p->use_tasks ? 1 : 0;
    // one staging buffer is enough when no multisplit pass runs (no levels, or one level done by the expansion)
    const int n_buf = prm.n_levels > (p->direct ? 1 : 0) ? 2 : 1;

    // ---- batches: consecutive heavy rows whose products fit one staging buffer.  Default size: a fifth of the
    // device's memory for staging (fewer, longer launches: on R-MAT scale 20, 2^31 products per batch instead of
    // 2^29 took 7 % off the step), at least 2^29 products, at most what 32-bit tile positions allow.
    i64 stage = p->opts.stage_elems;
    if (stage <= 0) {
      stage = std::max<i64>(i64{1} << 29, static_cast<i64>(facts.total_mem / 5) / (static_cast<i64>(n_buf) * (4 + p->sv)));
      stage = std::max(stage, info.products_max_row);  // a row is never split
    }
    stage = std::min(stage, info.products_heavy);
    const i64 kMaxStage = (i64{1} << 31) - kSplitTile;  // batch-relative positions are 32-bit in the multisplit tiles
    if (stage > kMaxStage) stage = kMaxStage;
    if (info.products_max_row > stage)
      return fail(GM_ERR_CAPACITY, "a heavy row has " + std::to_string(info.products_max_row) +
                                       " products, more than one staging half-buffer holds (" + std::to_string(stage) + ")");
    if (stage >= info.products_heavy) {  // everything at once: nothing to cut, the lists stay on the device
      p->batches.push_back(Batch{0, nH, 0, info.products_heavy});
    } else {
      std::vector<int64_t> hb(static_cast<size_t>(nH) + 1);
      p->x_heavy_host.resize(static_cast<size_t>(nH));
      p->heavy_nz_off_host.resize(static_cast<size_t>(nH) + 1);
      GM_CUDA(cudaMemcpyAsync(hb.data(), p->heavy_base, hb.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
      GM_CUDA(cudaMemcpyAsync(p->x_heavy_host.data(), p->x_heavy, static_cast<size_t>(nH) * sizeof(int32_t),
                              cudaMemcpyDeviceToHost, st));
      GM_CUDA(cudaMemcpyAsync(p->heavy_nz_off_host.data(), p->heavy_nz_off, (static_cast<size_t>(nH) + 1) * sizeof(int64_t),
                              cudaMemcpyDeviceToHost, st));
      GM_CUDA(cudaStreamSynchronize(st));
      if (!cut_batches(hb.data(), nH, stage, &p->batches)) return fail(GM_ERR_CAPACITY, "batch cutting failed");
    }
    info.n_batches = static_cast<int64_t>(p->batches.size());
    info.stage_elems = 0;
    for (const Batch& b : p->batches) {
      info.stage_elems = std::max(info.stage_elems, b.elems);
      p->max_batch_rows = std::max(p->max_batch_rows, b.h1 - b.h0);
    }
    // the accumulate kernel streams whole tiles: it may read (and ignore) up to one tile past the last product
    const size_t se = static_cast<size_t>(info.stage_elems) + 4096 + 8;
    for (int i = 0; i < n_buf; ++i) {
      GM_TRY(plan_alloc(p, &p->stage_col[i], se, st));
      unsigned char* v = nullptr;
      GM_TRY(plan_alloc(p, &v, se * static_cast<size_t>(p->sv), st));
      p->stage_val[i] = v;
    }
    if (p->use_tasks) {
      p->use_panels = plan_panel_rules(p);
      p->pending = true;  // (the lists' kernels may still run when the call returns: see gm_spgemm_execute)
      GM_TRY(plan_tasks(p, st));
      return GM_OK;
    }
    // ---- segment table: one segment per stored entry of a heavy row
    {
      i64* tmp2 = nullptr;
      int32_t* seg_len = nullptr;
      Arena ar;
      ar.add(&p->seg_off, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&p->seg_bstart, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&p->seg_j, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&p->seg_brow, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&p->seg_hrow, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&seg_len, static_cast<size_t>(p->n_seg) + 1);
      ar.add(&tmp2, static_cast<size_t>(scan_tmp_elems(p->n_seg)));
      GM_TRY(ar.commit(p, st));
      k1_heavy_segments<<<static_cast<unsigned>((p->n_seg + 8 * kSegRun - 1) / (8 * kSegRun)), 256, 0, st>>>(
          p->x_heavy, nH, p->heavy_nz_off, A.row_ptr, A.col_idx, B.row_ptr, p->n_seg, seg_len, p->seg_bstart, p->seg_j,
          p->seg_brow, p->seg_hrow);
      info.launches += 1 + exclusive_scan<int32_t, i64>(seg_len, p->seg_off, p->n_seg, tmp2, nullptr, nullptr, nullptr, st);
    }
    const size_t n_chunks_max = static_cast<size_t>(p->max_batch_rows) * static_cast<size_t>(prm.chunks_required);
    Arena ar;
    ar.add(&p->level_off[0], n_chunks_max + 1);
    if (prm.n_levels > 0) {
      ar.add(&p->counts, n_chunks_max + 1);
      ar.add(&p->cursor, n_chunks_max + 1);
      ar.add(&p->level_off[1], n_chunks_max + 1);
    }
    ar.add(&p->chunk_nnz, n_chunks_max + 1);
    ar.add(&p->chunk_nnz_off, n_chunks_max + 1);
    ar.add(&p->chunk_base, n_chunks_max + 1);
    ar.add(&p->mid_list, n_chunks_max + 1);
    ar.add(&p->big_list, n_chunks_max + 1);
    ar.add(&p->acc_counters, 8);
    if (p->exit_max >= 0) {
      ar.add(&p->exit_tag[0], n_chunks_max + 1);
      ar.add(&p->exit_tag[1], n_chunks_max + 1);
      ar.add(&p->parent_tag, n_chunks_max + 1);
    }
    const size_t n_tiles_max = static_cast<size_t>(info.stage_elems) / std::min({kExpandTileShort, kSplitTile, kGatherTileMin, kDirectTileSmall}) + 2;
    ar.add(&p->tile_meta, n_tiles_max);
    ar.add(&p->row_meta, n_tiles_max);
    i64 max_seg_b = 0;
    for (const Batch& b : p->batches) max_seg_b = std::max(max_seg_b, seg_begin(p, b.h1) - seg_begin(p, b.h0));
    if (p->direct) {
      const size_t F0 = static_cast<size_t>(prm.fanout[0]);
      ar.add(&p->child_bound, static_cast<size_t>(B.n_rows) * (F0 + 1) + 1);
      ar.add(&p->seg_prefix, (static_cast<size_t>(max_seg_b) + 1) * F0);
      ar.add(&p->seg_h, (static_cast<size_t>(max_seg_b) + 1) * F0);
      ar.add(&p->seg_tile_sums, (static_cast<size_t>(max_seg_b) / kGTile + 2) * F0);
      if (p->stream) ar.add(&p->seg_rec, (static_cast<size_t>(max_seg_b) + 1) * static_cast<size_t>(stream_rec_words(prm.fanout[0])));
    }
    i64 csc_scan_len = 0;
    if (p->csc) {
      ar.add(&p->csc_cnt, static_cast<size_t>(B.n_rows) + 1);
      ar.add(&p->csc_ptr, static_cast<size_t>(B.n_rows) + 2);
      ar.add(&p->csc_cursor, static_cast<size_t>(B.n_rows) + 2);
      ar.add(&p->csc_perm, static_cast<size_t>(max_seg_b) + 1);
      ar.add(&p->csc_len, static_cast<size_t>(max_seg_b) + 1);
      ar.add(&p->csc_off, static_cast<size_t>(max_seg_b) + 2);
      csc_scan_len = std::max<i64>(B.n_rows, max_seg_b);
    }
    // the per-batch scans can be longer than the ones above
    ar.add(&p->scan_tmp, static_cast<size_t>(scan_tmp_elems(std::max<i64>({static_cast<i64>(n_chunks_max), nA, csc_scan_len, 1}))));
    GM_TRY(ar.commit(p, st));
    if (p->direct && B.n_rows > 0) {
      k_child_bounds<<<grid_for(B.n_rows * (prm.fanout[0] + 1), 256, p->num_sms, 32), 256, 0, st>>>(
          B.row_ptr, B.col_idx, B.n_rows, prm.fanout[0], prm.shift[0], p->child_bound);
      ++info.launches;
    }
    p->pending = true;
  }
  return GM_OK;
}

// ------------------------------------------------------------------------------------------------
// execute
// ------------------------------------------------------------------------------------------------
template <typename V, bool NUMERIC, int G, int LPN, int BT>
static int launch_hash_one(gm_plan* p, const int32_t* rows, i64 n_rows, const int* n_rows_dev, int slots, int cap,
                           const i64* c_row_ptr, int32_t* c_col, V* c_val, i64 c_capacity, cudaStream_t st) {
  constexpr int kGroups = BT / G;
  const size_t smem = kGroups * light_group_bytes<V, NUMERIC>(slots, cap, G);
  constexpr auto kern = k3_light_rows<V, G, LPN, BT, NUMERIC>;
  // (static shared memory counts towards the 48 KB that need no opt-in)
  if (smem > 32 * 1024) GM_TRY(allow_smem<kern>(p));
  const unsigned grid = grid_for(n_rows, kGroups, p->num_sms, 2048 / BT * 4);
  kern<<<grid, BT, smem, st>>>(p->A.row_ptr, p->A.col_idx, static_cast<const V*>(p->A.vals), p->B.row_ptr, p->B.col_idx,
                               static_cast<const V*>(p->B.vals), rows, static_cast<int>(n_rows), n_rows_dev, slots, cap, p->row_nnz,
                               c_row_ptr, c_col, c_val, c_capacity, p->err);
  ++p->stats.launches;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// The hash accumulator's two passes (rows above kSortMaxProducts products).  Symbolic: the classes of the row analysis;
// numeric: the same rows binned again by their entry counts (n_rows: an upper bound, n_rows_dev: the bin's fill).
template <typename V, bool NUMERIC>
static int launch_hash(gm_plan* p, int cap, int slots, const int32_t* rows, i64 n_rows, const int* n_rows_dev,
                       const i64* c_row_ptr, int32_t* c_col, V* c_val, i64 c_capacity, cudaStream_t st) {
#define GM_LIGHT(G, LPN, BT) \
  launch_hash_one<V, NUMERIC, G, LPN, BT>(p, rows, n_rows, n_rows_dev, slots, cap, c_row_ptr, c_col, c_val, c_capacity, st)
  if (cap <= 16) return GM_LIGHT(8, 1, 256);
  if (cap <= 64) return GM_LIGHT(32, 4, 256);
  if (cap <= 256) return GM_LIGHT(128, 8, 128);
  if (cap <= 1024) return GM_LIGHT(256, 16, 256);
  if (cap <= 4096) return GM_LIGHT(512, 32, 512);
  return GM_LIGHT(1024, 32, 1024);
#undef GM_LIGHT
}

static RowSums row_sums_of(const gm_plan* p) {
  return p->row_sums ? RowSums{p->sums[p->sums_at], p->sums[p->sums_at ^ 1], row_sum_groups(p->A.n_rows)} : RowSums{nullptr, nullptr, 0};
}

// One thread per row: count, write to C, or write to the staging area.
template <typename V, int MODE>
static int launch_merge(gm_plan* p, const int32_t* rows, i64 n_rows, i64* c_row_ptr, int32_t* out_col, V* out_val,
                        cudaStream_t st) {
  const unsigned grid = static_cast<unsigned>((n_rows + kMergeThreads - 1) / kMergeThreads);
  // Entries for C are collected in shared memory, but the rows of B that neighbouring rows share want to stay in L1: with
  // 60 % of it as shared memory the 1024^2 grid's numeric pass takes 95 us, with all of it (more blocks per SM) 127, with 30 % 108.
#define GM_MERGE(NL)                                                                                                       \
  do {                                                                                                                     \
    auto kern = k3_merge_rows<V, NL, MODE>;                                                                                \
    if (MODE == kMergeToC || MODE == kMergePlace)                                                                          \
      GM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 60));                             \
    kern<<<grid, kMergeThreads, 0, st>>>(p->A.row_ptr, p->A.col_idx, static_cast<const V*>(p->A.vals), p->B.row_ptr,       \
                                         p->B.col_idx, static_cast<const V*>(p->B.vals), rows, n_rows, p->light_off,       \
                                         p->row_nnz, c_row_ptr, out_col, out_val, row_sums_of(p),                          \
                                         reinterpret_cast<i64*>(&p->slot->c_total));                                       \
  } while (0)
  // (an instance costs registers for the lists it has room for: the 1024^2 grid fp64, five lists, takes 254 us a call with the
  // instance for five, 279 with the one for eight)
  if (p->merge_lists <= 2) GM_MERGE(2);
  else if (p->merge_lists <= 4) GM_MERGE(4);
  else if (p->merge_lists <= 5) GM_MERGE(5);
  else GM_MERGE(kMergeMaxLists);
#undef GM_MERGE
  ++p->stats.launches;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

template <typename V, typename Key, int KMAX>
static int launch_sort_one(gm_plan* p, const SortLists& lists, i64 n, cudaStream_t st) {
  const unsigned grid = grid_for(n, kSortWarpsOf<KMAX>, p->num_sms, KMAX > 4 ? 16 : 24);
  k3_sort_rows<V, Key, KMAX><<<grid, kSortWarpsOf<KMAX> * 32, 0, st>>>(
      p->A.row_ptr, p->A.col_idx, static_cast<const V*>(p->A.vals), p->B.row_ptr, p->B.col_idx,
      static_cast<const V*>(p->B.vals), lists, p->light_off, p->row_nnz, p->light_col, static_cast<V*>(p->light_val), row_sums_of(p));
  ++p->stats.launches;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// Light rows, everything that does not need C: merged and sorted rows go to the staging area (when every row is merged
// they are only counted), hash rows are counted.
template <typename V>
static int light_front(gm_plan* p, cudaStream_t st) {
  const i64 stride = p->A.n_rows;
  auto list = [&](int c) { return p->class_list + static_cast<i64>(c) * stride; };
  if (p->merge_only)
    return launch_merge<V, kMergeCount>(p, nullptr, p->A.n_rows, nullptr, nullptr, nullptr, st);
  if (p->class_rows[kMergeClass] > 0)
    GM_TRY((launch_merge<V, kMergeToStage>(p, list(kMergeClass), p->class_rows[kMergeClass], nullptr, p->light_col,
                                           static_cast<V*>(p->light_val), st)));
  // a key packs a product's column with its position in the row: 32 bits unless the matrix is very wide
  int col_bits = 1;
  while (col_bits < 31 && (i64{1} << col_bits) < p->B.n_cols) ++col_bits;
  if (const i64 n = p->class_rows[kSortClass0 + 5]; n > 0) {
    SortLists l{};
    l.rows[0] = list(kSortClass0 + 5);
    l.n[0] = n;
    if (col_bits + 10 <= 32) GM_TRY((launch_sort_one<V, u32, 32>(p, l, n, st)));
    else GM_TRY((launch_sort_one<V, u64, 32>(p, l, n, st)));
  }
  {
    SortLists l{};
    for (int i = 0; i < 2; ++i) { const int c = kSortClass0 + 4 - i; l.rows[i] = list(c); l.n[i] = p->class_rows[c]; }
    SortLists wide{};  // rows whose keys take 64 bits
    for (int i = 0; i < 2; ++i)
      if (col_bits + 9 - i > 32) { wide.rows[i] = l.rows[i]; wide.n[i] = l.n[i]; l.n[i] = 0; }
    if (wide.n[0] + wide.n[1] > 0) GM_TRY((launch_sort_one<V, u64, 16>(p, wide, wide.n[0] + wide.n[1], st)));
    if (l.n[0] + l.n[1] > 0) GM_TRY((launch_sort_one<V, u32, 16>(p, l, l.n[0] + l.n[1], st)));
  }
  {
    SortLists l{};
    i64 n = 0;
    for (int i = 0; i < 3; ++i) { const int c = kSortClass0 + 2 - i; l.rows[i] = list(c); l.n[i] = p->class_rows[c]; n += l.n[i]; }
    if (n > 0 && col_bits + 7 <= 32) GM_TRY((launch_sort_one<V, u32, 4>(p, l, n, st)));
    else if (n > 0) GM_TRY((launch_sort_one<V, u64, 4>(p, l, n, st)));
  }
  for (int c = kHashClass0; c < kHashClass0 + p->rules.n_hash; ++c) {
    if (p->class_rows[c] <= 0) continue;
    const int cap = p->rules.hash_cap[c - kHashClass0];
    const int slots = cap == p->bins.cap[p->bins.n_bins - 1] ? p->bin_slots[p->bins.n_bins - 1] : 2 * cap;
    GM_TRY((launch_hash<V, false>(p, cap, slots, list(c), p->class_rows[c], nullptr, nullptr, nullptr, nullptr, 0, st)));
  }
  return GM_OK;
}

// Light rows [r0, r1) into C, once C.row_ptr covers them.
template <typename V>
static int light_back(gm_plan* p, i64 r0, i64 r1, i64* c_row_ptr, int32_t* c_col, V* c_val, i64 capacity, cudaStream_t st) {
  if (p->info.rows_light <= 0 || r1 <= r0) return GM_OK;
  if (p->merge_only && p->row_sums) return launch_merge<V, kMergePlace>(p, nullptr, p->A.n_rows, c_row_ptr, c_col, c_val, st);
  if (p->merge_only) return launch_merge<V, kMergeToC>(p, nullptr, p->A.n_rows, c_row_ptr, c_col, c_val, st);
  if (p->staged_light > 0) {
    i64 n_staged = 0;
    for (int c = 0; c < kHashClass0; ++c) n_staged += p->class_rows[c];
    const i64 avg = p->staged_light / n_staged;
#define GM_COPY(LPR)                                                                                                     \
  k3_copy_rows<V, LPR><<<static_cast<unsigned>(((r1 - r0) * LPR + 255) / 256), 256, 0, st>>>(                             \
      p->light_col, static_cast<const V*>(p->light_val), p->light_off, r0, r1, c_row_ptr, c_col, c_val, capacity, p->err)
#define GM_PLACE(LPR)                                                                                                             \
  k3_place_rows<V, LPR><<<static_cast<unsigned>((p->A.n_rows + kPlaceRows<LPR> - 1) / kPlaceRows<LPR>), 256, 0, st>>>(             \
      p->light_col, static_cast<const V*>(p->light_val), p->light_off, p->A.n_rows, p->row_nnz, row_sums_of(p), c_row_ptr, c_col, \
      c_val, capacity, reinterpret_cast<i64*>(&p->slot->c_total), p->err)
    if (p->row_sums) {  // (all rows: there are no batches)
      if (avg <= 16) GM_PLACE(8);
      else GM_PLACE(32);
    } else if (avg <= 16) GM_COPY(8);
    else GM_COPY(32);
#undef GM_COPY
#undef GM_PLACE
    ++p->stats.launches;
    GM_CUDA(cudaGetLastError());
  }
  if (p->num_rows) {
    GM_CUDA(cudaMemsetAsync(p->num_fill, 0, 8 * sizeof(int), st));
    k1_bin_rows<<<static_cast<unsigned>((r1 - r0 + 255) / 256), 256, 0, st>>>(
        p->row_nnz, p->heavy_flag, p->light_off, r0, r1 - r0, p->bins, p->A.n_rows, p->num_fill, p->num_rows);
    ++p->stats.launches;
    i64 upper = 0;  // a row's numeric bin is never above its class
    for (int c = kHashClass0; c < kRowClasses; ++c) upper += p->class_rows[c];
    for (int b = 0; b < p->bins.n_bins; ++b)
      GM_TRY((launch_hash<V, true>(p, p->bins.cap[b], p->bin_slots[b], p->num_rows + static_cast<i64>(b) * p->A.n_rows, upper,
                                   p->num_fill + b, c_row_ptr, c_col, c_val, capacity, st)));
  }
  return GM_OK;
}

__global__ void k_heavy_row_counts(const i64* __restrict__ chunk_nnz_off, int log2_chunks_per_row, i64 n_rows_b,
                                   const int32_t* __restrict__ x_heavy, i64 h0, int32_t* __restrict__ row_nnz,
                                   i64* __restrict__ heavy_total) {
  if (blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(reinterpret_cast<u64*>(heavy_total), static_cast<u64>(chunk_nnz_off[n_rows_b << log2_chunks_per_row]));
  for (i64 r = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; r < n_rows_b;
       r += static_cast<i64>(gridDim.x) * blockDim.x) {
    row_nnz[x_heavy[h0 + r]] =
        static_cast<int32_t>(chunk_nnz_off[(r + 1) << log2_chunks_per_row] - chunk_nnz_off[r << log2_chunks_per_row]);
  }
}

__global__ void k_rebase(const i64* __restrict__ in, i64 n, i64 bias, i64* __restrict__ out) {
  for (i64 i = static_cast<i64>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<i64>(gridDim.x) * blockDim.x)
    out[i] = in[i] - bias;
}

template <typename V>
struct HeavyBatchState {
  int32_t* fin_col = nullptr;  // staging buffer that holds the final chunks
  V* fin_val = nullptr;
  const i64* chunk_off = nullptr;    // n_chunks + 1 batch-relative offsets
  i64 n_chunks = 0;
  int log2_cpr = 0;
  // chunks that left the multisplit hierarchy early (tags == nullptr: none can have)
  const unsigned char* tags = nullptr;
  int32_t* alt_col = nullptr;  // the staging buffer that is not fin_col
  V* alt_val = nullptr;
  ExitTags xt;
};

// K6: accumulate every chunk of the batch and compact it in place; chunk_nnz receives the entry counts.
// Three kernels, one per size class of the chunks (see gm_k6_accumulate.cuh).
template <typename V>
static int launch_accumulate(gm_plan* p, const Batch& b, const HeavyBatchState<V>& hs, cudaStream_t st) {
  const gm_params& prm = p->info.params;
  const int W = prm.chunk_width;
  const int bt = prm.acc_block_threads;
  const int small_max = p->small_max, mid_max = p->mid_max;
  GM_CUDA(cudaMemsetAsync(p->acc_counters, 0, 8 * sizeof(int), st));
  GM_CUDA(cudaMemsetAsync(p->chunk_nnz, 0, static_cast<size_t>(hs.n_chunks) * sizeof(u32), st));
  if (p->opts.validate_inputs) {
    k6_validate_chunks<<<grid_for(hs.n_chunks * 32, 256, p->num_sms, 8), 256, 0, st>>>(
        hs.fin_col, hs.chunk_off, hs.n_chunks, hs.log2_cpr, W, p->B.n_cols, p->err, hs.tags, hs.alt_col, hs.xt);
    ++p->stats.launches;
  }
  k6_classify<<<grid_for(hs.n_chunks, 256, p->num_sms), 256, 0, st>>>(hs.chunk_off, hs.n_chunks, small_max, mid_max, p->mid_list,
                                                                     p->big_list, p->acc_counters);
  ++p->stats.launches;
  if (small_max > 0) {
    p->times.begin(PhaseTimes::kAccSmall, st);
    // as many blocks as are resident at once: the warps share out the chunks statically, so a block that had to wait
    // for a free slot would start its share when the others are done
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k6_small_chunks<V>, kSmallWarps * 32, 0) != cudaSuccess || per_sm < 1)
      per_sm = 4;
    k6_small_chunks<V><<<static_cast<unsigned>(p->num_sms * per_sm), kSmallWarps * 32, 0, st>>>(
        hs.fin_col, hs.fin_val, hs.chunk_off, hs.n_chunks,
        std::max(0, std::min(hs.log2_cpr, 32 - kSmallIdxBits - ilog2_floor(static_cast<uint64_t>(W)))), small_max, p->chunk_nnz,
        reinterpret_cast<u64*>(p->c_total + 2), hs.tags, hs.alt_col, hs.alt_val, hs.xt);
    ++p->stats.launches;
    p->times.end(st);
  }
  if (mid_max > small_max) {
    p->times.begin(PhaseTimes::kAccMid, st);
    const size_t smem = mid_smem_bytes(W, sizeof(V), mid_max);
    constexpr auto kern = k6_mid_chunks<V>;
    if (smem > 32 * 1024) GM_TRY(allow_smem<kern>(p));
    const int per_sm = std::max<int>(1, std::min<int>(2048 / kMidThreads, static_cast<int>((p->smem_bytes - 1024) / (smem + 1024))));
    const unsigned grid = static_cast<unsigned>(std::min<i64>(hs.n_chunks, static_cast<i64>(p->num_sms) * per_sm));
    kern<<<grid, kMidThreads, smem, st>>>(hs.fin_col, hs.fin_val, hs.chunk_off, p->mid_list, p->acc_counters, hs.log2_cpr, W,
                                          mid_max, p->chunk_nnz, reinterpret_cast<u64*>(p->c_total + 4));
    ++p->stats.launches;
    p->times.end(st);
  }
  p->times.begin(PhaseTimes::kAccNum, st);
  {
    const size_t smem = acc_smem_bytes_big(W, sizeof(V));
    const int per_sm = 1024 / bt;
    const unsigned grid = static_cast<unsigned>(std::min<i64>(hs.n_chunks, static_cast<i64>(p->num_sms) * per_sm));
#define GM_ACC(BT)                                                                                                   \
  do {                                                                                                               \
    constexpr auto kern = k6_accumulate<V, BT>;                                                                      \
    if (smem > 32 * 1024) GM_TRY(allow_smem<kern>(p));                                                               \
    kern<<<grid, BT, smem, st>>>(hs.fin_col, hs.fin_val, hs.chunk_off, hs.n_chunks, p->big_list, p->acc_counters,    \
                                 hs.log2_cpr, W, p->chunk_nnz);                                                      \
  } while (0)
    if (bt == 1024) GM_ACC(1024);
    else if (bt == 512) GM_ACC(512);
    else if (bt == 256) GM_ACC(256);
    else GM_ACC(128);
#undef GM_ACC
  }
  p->times.end(st);
  ++p->stats.launches;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// K7: once C.rowPtr covers the batch's rows, move the compacted chunks into C.
template <typename V>
static int launch_gather(gm_plan* p, const Batch& b, const HeavyBatchState<V>& hs, const i64* c_row_ptr,
                         int32_t* c_col, V* c_val, i64 c_capacity, cudaStream_t st) {
  k6_chunk_bases<<<grid_for(hs.n_chunks, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, hs.n_chunks, hs.log2_cpr,
                                                                         p->x_heavy, b.h0, c_row_ptr, p->chunk_base);
  // the batch's heavy entry count is only known on the device: it is at most the batch's product count
  const int tile = gather_tile(hs.n_chunks, b.elems);
  const unsigned grid = static_cast<unsigned>((b.elems + tile - 1) / tile);
  k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, hs.n_chunks, 0, 0, tile, p->tile_meta,
                                                               p->chunk_nnz_off + hs.n_chunks);
  const bool alt = hs.tags && hs.xt.alt_bits;
  const unsigned most = static_cast<unsigned>(p->num_sms * kGatherBlocksPerSm);
#define GM_GATHER(ALT, LOOP) \
  (tile == kGatherTile ? k7_gather<V, kGatherTile, ALT, LOOP> : tile == 4096 ? k7_gather<V, 4096, ALT, LOOP> : k7_gather<V, 2048, ALT, LOOP>)
  auto kern = grid > most ? (alt ? GM_GATHER(true, true) : GM_GATHER(false, true)) : (alt ? GM_GATHER(true, false) : GM_GATHER(false, false));
#undef GM_GATHER
  kern<<<std::min(grid, most), kGatherThreads, 0, st>>>(hs.fin_col, hs.fin_val, hs.chunk_off, p->chunk_nnz_off, p->chunk_base, hs.n_chunks,
                                        p->tile_meta, c_col, c_val, c_capacity, p->err, alt ? hs.alt_col : nullptr,
                                        alt ? hs.alt_val : nullptr, alt ? hs.tags : nullptr, alt ? hs.xt.alt_bits : 0);
  p->stats.launches += 3;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// Expansion, every multisplit level and the accumulate of one batch.  Leaves the compacted chunks in
// the staging buffer and the per-chunk entry counts (and their scan) in chunk_nnz / chunk_nnz_off,
// and writes the heavy rows' entry counts into row_nnz.
template <typename V>
static int heavy_batch_front(gm_plan* p, const Batch& b, HeavyBatchState<V>* hs, cudaStream_t st) {
  const gm_params& prm = p->info.params;
  const i64 rows_b = b.h1 - b.h0;
  PhaseTimes& tm = p->times;
  // level-0 parents are the batch's rows: offsets relative to the batch
  i64* off_cur = p->level_off[0];
  i64* off_nxt = p->level_off[1];
  k_rebase<<<grid_for(rows_b + 1, 256, p->num_sms), 256, 0, st>>>(p->heavy_base + b.h0, rows_b + 1, b.elem0, off_cur);
  ++p->stats.launches;
  int cur = 0;
  i64 n_par = rows_b;
  int first_level = 0;
  if (p->direct) {
    // ---- run starts of every (segment, child) from counts alone, then the products straight into the children
    const int F = prm.fanout[0];
    const i64 seg0 = seg_begin(p, b.h0);
    const i64 n_seg_b = seg_begin(p, b.h1) - seg0;
    const i64 n_gt = (n_seg_b + kGTile - 1) / kGTile;
    const i64 n_child = rows_b * F;
    const unsigned ggrid = static_cast<unsigned>((n_gt + (256 / F) - 1) / (256 / F));
    tm.begin(PhaseTimes::kHist, st);
    k_g_tile_sums<<<ggrid, 256, 0, st>>>(p->seg_brow, seg0, n_seg_b, p->child_bound, F, p->seg_tile_sums);
    k_g_scan_tiles<<<static_cast<unsigned>(F), 256, 0, st>>>(p->seg_tile_sums, n_gt, F);
    k_g_write<<<ggrid, 256, 0, st>>>(p->seg_brow, seg0, n_seg_b, p->child_bound, F, p->seg_tile_sums, p->seg_prefix, p->seg_h);
    k_g_row_counts<<<grid_for(n_child, 256, p->num_sms, 32), 256, 0, st>>>(p->seg_prefix, p->heavy_nz_off + b.h0, seg0, rows_b, F,
                                                                          p->counts);
    p->stats.launches += 4;
    tm.end(st);
    tm.begin(PhaseTimes::kScan, st);
    p->stats.launches += 1 + exclusive_scan<u32, i64>(p->counts, off_nxt, n_child, p->scan_tmp, nullptr, nullptr, nullptr, st);
    // (the cursor array of the multisplit is free in this mode: it holds R)
    u32* const row_base = reinterpret_cast<u32*>(p->cursor);
    k_g_row_base<<<grid_for(n_child, 256, p->num_sms, 32), 256, 0, st>>>(p->seg_prefix, p->heavy_nz_off + b.h0, seg0, rows_b, F,
                                                                        off_nxt, row_base);
    tm.end(st);
    tm.begin(PhaseTimes::kExpand, st);
    if (p->stream) {
      // one contiguous range of the batch's products per warp; the grid fills the SMs' shared memory
      const size_t smem = kStreamWarps * stream_warp_smem_bytes(F, sizeof(V));
      const int per_sm = std::max<int>(1, std::min<int>(16, static_cast<int>((p->smem_bytes - 1024) / (smem + 1024))));
      const i64 n_warps = static_cast<i64>(p->num_sms) * per_sm * kStreamWarps;
      const i64 per_warp = std::max<i64>(4096, ((b.elems + n_warps - 1) / n_warps + 127) & ~i64{127});
      const i64 n_ranges = (b.elems + per_warp - 1) / per_warp;
      const unsigned grid = static_cast<unsigned>((n_ranges + kStreamWarps - 1) / kStreamWarps);
      k_seg_records<V><<<grid_for(n_seg_b * stream_rec_words(F), 256, p->num_sms, 32), 256, 0, st>>>(
          p->seg_h, row_base, p->seg_hrow, p->seg_j, static_cast<const V*>(p->A.vals), seg0, n_seg_b, b.h0, F, p->seg_rec);
      k_tile_bounds<<<grid_for(n_ranges, 256, p->num_sms), 256, 0, st>>>(p->seg_off, p->n_seg, b.elem0, b.elems,
                                                                       static_cast<int>(per_warp), p->tile_meta);
      constexpr auto kern = k4_expand_stream<V>;
      GM_TRY(allow_smem<kern>(p));
      const int spin = p->opts.debug_spin_limit != 0 ? p->opts.debug_spin_limit : kCopySpinLimit;
      kern<<<grid, kStreamWarps * 32, smem, st>>>(p->seg_off, p->seg_bstart, p->n_seg, p->tile_meta, p->B.col_idx,
                                                  static_cast<const V*>(p->B.vals), p->B.nnz, b.elem0, b.elems, per_warp, seg0,
                                                  p->seg_rec, F, prm.shift[0], p->stage_col[0], static_cast<V*>(p->stage_val[0]),
                                                  spin, p->err);
      k4_expand_short<V><<<grid_for(n_seg_b * 32, 256, p->num_sms, 8), 256, 0, st>>>(
          p->seg_off, p->seg_bstart, p->B.col_idx, static_cast<const V*>(p->B.vals), seg0, n_seg_b, p->seg_rec, F, prm.shift[0],
          p->stage_col[0], static_cast<V*>(p->stage_val[0]));
    } else {
      const int tile = direct_tile(F);
      const unsigned grid = static_cast<unsigned>((b.elems + tile - 1) / tile);
      k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(p->seg_off, p->n_seg, b.elem0, b.elems, tile, p->tile_meta);
      k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(off_cur, rows_b, 0, b.elems, tile, p->row_meta);
      auto kern = tile == kDirectTileSmall ? k4_expand_direct<V, kDirectTileSmall> : k4_expand_direct<V, kExpandTile>;
      kern<<<grid, kExpandThreads, 0, st>>>(
          p->seg_off, p->seg_bstart, p->seg_j, p->tile_meta, static_cast<const V*>(p->A.vals), p->B.col_idx,
          static_cast<const V*>(p->B.vals), b.elem0, b.elems, p->row_meta, off_cur, seg0, F, prm.shift[0], row_base, p->seg_h,
          p->stage_col[0], static_cast<V*>(p->stage_val[0]));
    }
    p->stats.launches += 3;
    GM_CUDA(cudaGetLastError());
    tm.end(st);
    std::swap(off_cur, off_nxt);
    n_par = n_child;
    first_level = 1;
  }
  // the expansion kernel counts the first level's (row, child) bins while it writes, unless asked not to
  const bool fuse_hist = !p->direct && prm.n_levels > 0 && !p->opts.separate_histogram && !p->csc;
  if (p->csc) {
    // ---- outer-product order: masked CSR -> CSC of the batch's segments (counting sort by row of B), then the
    // expansion walks the product space in that order
    tm.begin(PhaseTimes::kExpand, st);
    const i64 seg0 = seg_begin(p, b.h0);
    const i64 n_seg_b = seg_begin(p, b.h1) - seg0;
    const i64 nB = p->B.n_rows;
    GM_CUDA(cudaMemsetAsync(p->csc_cnt, 0, static_cast<size_t>(nB + 1) * sizeof(int32_t), st));
    k_csc_count<<<grid_for(n_seg_b, 256, p->num_sms, 16), 256, 0, st>>>(p->seg_brow, seg0, n_seg_b, p->csc_cnt);
    exclusive_scan<int32_t, i64>(p->csc_cnt, p->csc_ptr, nB, p->scan_tmp, nullptr, nullptr, reinterpret_cast<i64*>(p->csc_cursor), st);
    k_csc_scatter<<<grid_for(n_seg_b, 256, p->num_sms, 16), 256, 0, st>>>(p->seg_brow, p->seg_off, seg0, n_seg_b, p->csc_cursor,
                                                                          p->csc_perm, p->csc_len);
    exclusive_scan<int32_t, i64>(p->csc_len, p->csc_off, n_seg_b, p->scan_tmp, nullptr, nullptr, nullptr, st);
    const unsigned grid = static_cast<unsigned>((b.elems + kExpandTile - 1) / kExpandTile);
    k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(p->csc_off, n_seg_b, 0, b.elems, kExpandTile, p->tile_meta);
    k4_expand_csc<V><<<grid, kExpandThreads, 0, st>>>(p->csc_off, p->csc_perm, p->seg_off, p->seg_bstart, p->seg_j, seg0,
                                                      p->tile_meta, static_cast<const V*>(p->A.vals), p->B.col_idx,
                                                      static_cast<const V*>(p->B.vals), b.elem0, b.elems, p->stage_col[0],
                                                      static_cast<V*>(p->stage_val[0]));
    p->stats.launches += 10;
    GM_CUDA(cudaGetLastError());
    tm.end(st);
  } else if (!p->direct) {
  tm.begin(PhaseTimes::kExpand, st);
  {
    const bool short_segments = p->info.products_heavy < kExpandShortSegment * p->n_seg;
    const int tile = short_segments ? kExpandTileShort : kExpandTile;
    const unsigned grid = static_cast<unsigned>((b.elems + tile - 1) / tile);
    k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(p->seg_off, p->n_seg, b.elem0, b.elems, tile, p->tile_meta);
    ++p->stats.launches;
    if (fuse_hist) {
      GM_CUDA(cudaMemsetAsync(p->counts, 0, static_cast<size_t>(rows_b) * prm.fanout[0] * sizeof(u32), st));
      k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(off_cur, rows_b, 0, b.elems, tile, p->row_meta);
      ++p->stats.launches;
    }
    auto kern = short_segments ? k4_expand<V, kExpandTileShort> : k4_expand<V, kExpandTile>;
    kern<<<grid, kExpandThreads, 0, st>>>(p->seg_off, p->seg_bstart, p->seg_j, p->tile_meta,
                                                  static_cast<const V*>(p->A.vals), p->B.col_idx,
                                                  static_cast<const V*>(p->B.vals), b.elem0, b.elems, p->stage_col[0],
                                                  static_cast<V*>(p->stage_val[0]), p->row_meta, off_cur,
                                                  fuse_hist ? prm.fanout[0] : 0, fuse_hist ? prm.shift[0] : 0, p->counts);
    ++p->stats.launches;
    GM_CUDA(cudaGetLastError());
  }
  tm.end(st);
  }
  if (prm.n_levels > first_level) {
    GM_CUDA(cudaFuncSetAttribute(k5_level<V, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(split_smem_bytes<V>(true))));
    GM_CUDA(cudaFuncSetAttribute(k5_level<V, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(split_smem_bytes<V>(true))));
    GM_CUDA(cudaFuncSetAttribute(k5_level<V, true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(split_smem_bytes<V>(true))));
    GM_CUDA(cudaFuncSetAttribute(k5_level<V, true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(split_smem_bytes<V>(true))));
  }
  bool hist_ready = false;  // the previous level's multisplit counted this level's bins while it wrote
  // early exit: tags of the current parents (none before the first level that can leave chunks behind)
  const unsigned char* tag_cur = nullptr;
  int tag_buf = 0;
  int level_buf[GM_MAX_LEVELS + 1] = {0};  // staging buffer a level read from
  for (int l = first_level; l < prm.n_levels; ++l) {
    const int F = prm.fanout[l];
    const i64 n_child = n_par * F;
    const unsigned grid = static_cast<unsigned>((b.elems + kSplitTile - 1) / kSplitTile);
    const int32_t* xc = p->stage_col[cur];
    const V* xv = static_cast<const V*>(p->stage_val[cur]);
    tm.begin(PhaseTimes::kHist, st);
    k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(off_cur, n_par, 0, b.elems, kSplitTile, p->tile_meta);
    ++p->stats.launches;
    if (!(l == 0 && fuse_hist) && !hist_ready) {
      GM_CUDA(cudaMemsetAsync(p->counts, 0, static_cast<size_t>(n_child) * sizeof(u32), st));
      k5_level<V, false><<<grid, kSplitThreads, split_smem_bytes<V>(false), st>>>(
          xc, xv, b.elems, off_cur, n_par, p->tile_meta, F, prm.shift[l], p->counts, nullptr, nullptr, nullptr, 0, 0, nullptr);
      ++p->stats.launches;
      GM_CUDA(cudaGetLastError());
    }
    // Early exit: a parent of a level after the first that holds few products stays where it is; its span of columns
    // must still fit the sort's packed key
    level_buf[l] = cur;
    const int span_bits = prm.shift[l] + ilog2_floor(static_cast<uint64_t>(F));
    const bool can_exit = p->exit_max >= 0 && l >= 1 && span_bits + kSmallIdxBits <= 32;
    const bool exiting = can_exit || tag_cur != nullptr;
    if (exiting) {
      unsigned char* tag_nxt = p->exit_tag[tag_buf];
      k5_exit_flags<<<grid_for(n_child, 256, p->num_sms, 32), 256, 0, st>>>(
          off_cur, n_par, ilog2_floor(static_cast<uint64_t>(F)), tag_cur, can_exit ? p->exit_max : -1, l + 1, p->counts,
          p->parent_tag, tag_nxt, reinterpret_cast<u64*>(p->c_total + 6));
      ++p->stats.launches;
      tag_cur = tag_nxt;
      tag_buf ^= 1;
      hs->xt.set(l + 1, false, span_bits);  // (which buffer: known once the last level has run)
    }
    tm.end(st);
    tm.begin(PhaseTimes::kScan, st);
    p->stats.launches +=
        exclusive_scan<u32, i64>(p->counts, off_nxt, n_child, p->scan_tmp, nullptr, nullptr, reinterpret_cast<i64*>(p->cursor), st);
    tm.end(st);
    tm.begin(PhaseTimes::kSplit, st);
    // the counts of this level have been scanned: the array is free to receive the next level's
    const bool next = l + 1 < prm.n_levels && !p->opts.separate_histogram;
    if (next) GM_CUDA(cudaMemsetAsync(p->counts, 0, static_cast<size_t>(n_child) * prm.fanout[l + 1] * sizeof(u32), st));
    if (exiting && next) {
      k5_level<V, true, true, true><<<grid, kSplitThreads, split_smem_bytes<V>(true), st>>>(
          xc, xv, b.elems, off_cur, n_par, p->tile_meta, F, prm.shift[l], nullptr, p->cursor, p->stage_col[cur ^ 1],
          static_cast<V*>(p->stage_val[cur ^ 1]), prm.fanout[l + 1], prm.shift[l + 1], p->counts, p->parent_tag);
    } else if (exiting) {
      k5_level<V, true, false, true><<<grid, kSplitThreads, split_smem_bytes<V>(true), st>>>(
          xc, xv, b.elems, off_cur, n_par, p->tile_meta, F, prm.shift[l], nullptr, p->cursor, p->stage_col[cur ^ 1],
          static_cast<V*>(p->stage_val[cur ^ 1]), 0, 0, nullptr, p->parent_tag);
    } else if (next) {
      k5_level<V, true, true><<<grid, kSplitThreads, split_smem_bytes<V>(true), st>>>(
          xc, xv, b.elems, off_cur, n_par, p->tile_meta, F, prm.shift[l], nullptr, p->cursor, p->stage_col[cur ^ 1],
          static_cast<V*>(p->stage_val[cur ^ 1]), prm.fanout[l + 1], prm.shift[l + 1], p->counts);
    } else {
      k5_level<V, true, false><<<grid, kSplitThreads, split_smem_bytes<V>(true), st>>>(
          xc, xv, b.elems, off_cur, n_par, p->tile_meta, F, prm.shift[l], nullptr, p->cursor, p->stage_col[cur ^ 1],
          static_cast<V*>(p->stage_val[cur ^ 1]), 0, 0, nullptr);
    }
    p->stats.split_products += b.elems;
    hist_ready = next;
    ++p->stats.launches;
    GM_CUDA(cudaGetLastError());
    tm.end(st);
    std::swap(off_cur, off_nxt);
    cur ^= 1;
    n_par = n_child;
  }
  hs->fin_col = p->stage_col[cur];
  hs->fin_val = static_cast<V*>(p->stage_val[cur]);
  hs->chunk_off = off_cur;
  hs->n_chunks = n_par;
  hs->log2_cpr = ilog2_floor(static_cast<uint64_t>(prm.chunks_required));
  hs->tags = tag_cur;
  if (tag_cur) {
    hs->alt_col = p->stage_col[cur ^ 1];
    hs->alt_val = static_cast<V*>(p->stage_val[cur ^ 1]);
    for (int l = 1; l < prm.n_levels; ++l)
      if (level_buf[l] != cur) hs->xt.alt_bits |= 1u << (l + 1);
  }
  p->stats.final_chunks += n_par;
  p->stats.staged_products += b.elems;

  GM_TRY((launch_accumulate<V>(p, b, *hs, st)));  // (records its own two phases)
  tm.begin(PhaseTimes::kScan, st);
  p->stats.launches +=
      1 + exclusive_scan<u32, i64>(p->chunk_nnz, p->chunk_nnz_off, hs->n_chunks, p->scan_tmp, nullptr, nullptr, nullptr, st);
  k_heavy_row_counts<<<grid_for(rows_b, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, hs->log2_cpr, rows_b, p->x_heavy,
                                                                        b.h0, p->row_nnz, p->c_total + 1);
  tm.end(st);
  return GM_OK;
}

static int dev_error_to_status(int code) {
  switch (code) {
    case kDevOk: return GM_OK;
    case kDevCapacity: return fail(GM_ERR_CAPACITY, "C did not fit the room reserved for it (raise c_capacity or stage fewer products)");
    case kDevTableFull: return fail(GM_ERR_INTERNAL, "a light-row hash table overflowed");
    case kDevBadChunk: return fail(GM_ERR_INTERNAL, "an intermediate product reached a chunk that does not own its column");
    case kDevTimeout: return fail(GM_ERR_TIMEOUT, "a bounded wait on an asynchronous copy gave up");
    default: return fail(GM_ERR_INTERNAL, "unknown device error code");
  }
}

template <typename V>
static TaskInput<V> task_input(const gm_plan* p) {
  return TaskInput<V>{p->A.col_idx, static_cast<const V*>(p->A.vals), p->B.col_idx, static_cast<const V*>(p->B.vals),
                      p->piece_bound, p->task_rules.granules, p->task_rules.log2_g};
}

// Debug mode: nothing is summed when a product is not in the columns of its task (the sums keep a task's columns in shared memory).
template <typename V>
static int validate_tasks(gm_plan* p, cudaStream_t st) {
  k_validate_tasks<V><<<grid_for(p->info.rows_heavy, 1, p->num_sms, 8), 256, 0, st>>>(task_input<V>(p), p->tasks, p->row_task_off, p->heavy_base,
                                                                                    p->info.rows_heavy, p->B.n_cols, p->err);
  ++p->stats.launches;
  if (p->use_panels) {
    k_validate_panels<<<static_cast<unsigned>(p->num_sms * 4), 256, 0, st>>>(p->panels, p->x_heavy, p->info.rows_heavy, p->heavy_base, p->heavy_nz_off,
                                                                            p->A.row_ptr, p->A.col_idx, p->B.row_ptr, p->B.col_idx, p->B.n_rows,
                                                                            p->B.n_cols, panel_group_bits(p->sv), p->err);
    ++p->stats.launches;
  }
  GM_CUDA(cudaGetLastError());
  GM_CUDA(cudaStreamSynchronize(st));
  return dev_error_to_status(*static_cast<volatile int*>(&p->slot->err[0]));
}

// The tasks of one batch: sums into the staging area.  BIG: the dense accumulator's tasks, else the other classes (on the
// second stream: their blocks fill the SMs as the last big tasks run out).
template <typename V, bool BIG>
static int task_batch_sums(gm_plan* p, size_t bi, cudaStream_t st) {
  const Batch& b = p->batches[bi];
  const TaskRules& r = p->task_rules;
  const i64 t0 = p->task_begin[bi], n = p->task_begin[bi + 1] - t0;
  const HeavyTask* tasks = p->tasks + t0;
  const int* counters = p->task_counters + 8 * bi;
  int* tickets = p->task_tickets + 4 * bi;
  int32_t* out_col = p->stage_col[0];
  V* out_val = static_cast<V*>(p->stage_val[0]);
  const TaskInput<V> in = task_input<V>(p);
  PhaseTimes& tm = p->times;
  if constexpr (BIG) {
    tm.begin(PhaseTimes::kAccNum, st);
    if (p->use_panels) {
      constexpr auto kern = k6_panels<V>;
      GM_TRY(allow_smem<kern>(p));
      kern<<<static_cast<unsigned>(p->num_sms * 2), kPanelThreads, sizeof(PanelSmem<V>), st>>>(
          p->A.row_ptr, static_cast<const V*>(p->A.vals), static_cast<const V*>(p->B.vals), p->panels, p->x_heavy, p->heavy_base,
          p->heavy_nz_off, b.h0, b.h1, b.elem0, p->row_task_off, tickets + 2, out_col, out_val, p->chunk_nnz,
          reinterpret_cast<u64*>(p->c_total + 9));
      ++p->stats.launches;
    }
    const size_t smem = big_task_smem_bytes<V>(p->acc_width, p->acc_threads);
    const unsigned grid = static_cast<unsigned>(std::min<i64>(n, static_cast<i64>(p->num_sms) * p->acc_blocks));
#define GM_BIG(BT, BLOCKS)                                                                                                        \
  do {                                                                                                                    \
    constexpr auto kern = k6_big_tasks<V, BT, BLOCKS>;                                                                    \
    GM_TRY(allow_smem<kern>(p));                                                                                          \
    kern<<<grid, BT, smem, st>>>(in, tasks, n, p->task_list[2] + t0, counters, tickets, out_col, out_val, p->chunk_nnz);  \
  } while (0)
    if (p->acc_blocks == kBigBlocks && p->acc_threads == kBigThreads) GM_BIG(kBigThreads, kBigBlocks);
    else if (p->acc_blocks == 1) GM_BIG(1024, 1);
    else if (p->acc_blocks == 2) GM_BIG(512, 2);
    else if (p->acc_blocks == 4) GM_BIG(256, 4);
    else GM_BIG(128, 8);
#undef GM_BIG
    ++p->stats.launches;
    tm.end(st);
    GM_CUDA(cudaGetLastError());
    return GM_OK;
  }
  if (r.mid_max > r.small_max) {
    tm.begin(PhaseTimes::kAccMid, st);
    const size_t smem = mid_task_smem_bytes(static_cast<int>(r.mid_width), sizeof(V), r.mid_max);
    constexpr auto kern = k6_mid_tasks<V>;
    GM_TRY(allow_smem<kern>(p));
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMidThreads, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
    kern<<<static_cast<unsigned>(std::min<i64>(n, static_cast<i64>(p->num_sms) * per_sm)), kMidThreads, smem, st>>>(
        in, tasks, p->task_list[1] + t0, counters + 1, tickets + 1, static_cast<int>(r.mid_width), r.mid_max, out_col, out_val, p->chunk_nnz,
        reinterpret_cast<u64*>(p->c_total + 4));
    ++p->stats.launches;
    tm.end(st);
  }
  if (r.small_max > 0) {
    tm.begin(PhaseTimes::kAccSmall, st);
    const unsigned grid = static_cast<unsigned>(std::min<i64>((n + kSmallWarps - 1) / kSmallWarps, static_cast<i64>(p->num_sms) * (r.small_max > 128 ? 8 : 10)));
    if (r.small_max > 128)
      k6_small_tasks<V, 16><<<grid, kSmallWarps * 32, 0, st>>>(in, tasks, p->task_list[0] + t0, counters, out_col, out_val, p->chunk_nnz,
                                                             reinterpret_cast<u64*>(p->c_total + 2));
    else
      k6_small_tasks<V, 4><<<grid, kSmallWarps * 32, 0, st>>>(in, tasks, p->task_list[0] + t0, counters, out_col, out_val, p->chunk_nnz,
                                                            reinterpret_cast<u64*>(p->c_total + 2));
    ++p->stats.launches;
    tm.end(st);
  }
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// Prefix sums of the batch's entry counts, entries per heavy row.
static int task_batch_counts(gm_plan* p, size_t bi, cudaStream_t st) {
  const Batch& b = p->batches[bi];
  const i64 n = p->task_begin[bi + 1] - p->task_begin[bi];
  PhaseTimes& tm = p->times;
  tm.begin(PhaseTimes::kScan, st);
  p->stats.launches += 1 + exclusive_scan<u32, i64>(p->chunk_nnz, p->chunk_nnz_off, n, p->scan_tmp, nullptr, nullptr, nullptr, st);
  k_task_row_counts<<<grid_for(b.h1 - b.h0, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, p->row_task_off, b.h0, b.h1, p->x_heavy,
                                                                          p->row_nnz, p->c_total + 1);
  tm.end(st);
  p->stats.final_chunks += (b.h1 - b.h0) * p->info.params.chunks_required;
  p->stats.staged_products += b.elems;
  return GM_OK;
}

template <typename V>
static int task_batch_gather(gm_plan* p, size_t bi, bool bases, const i64* c_row_ptr, int32_t* c_col, V* c_val, i64 c_capacity, cudaStream_t st) {
  const Batch& b = p->batches[bi];
  const i64 t0 = p->task_begin[bi], n = p->task_begin[bi + 1] - t0;
  // the batch's entry count is only known on the device: it is at most the batch's product count
  const unsigned grid = static_cast<unsigned>((b.elems + kGatherTile - 1) / kGatherTile);
  if (bases) {
    k_task_bases<<<grid_for(b.h1 - b.h0, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, p->row_task_off, b.h0, b.h1, p->x_heavy, c_row_ptr,
                                                                       p->chunk_base);
    k_tile_bounds<<<grid_for(grid, 256, p->num_sms), 256, 0, st>>>(p->chunk_nnz_off, n, 0, 0, kGatherTile, p->tile_meta, p->chunk_nnz_off + n);
    p->stats.launches += 2;
  }
  k7_gather<V, kGatherTile><<<std::min(grid, static_cast<unsigned>(p->num_sms * kGatherBlocksPerSm)), kGatherThreads, 0, st>>>(
      p->stage_col[0], static_cast<const V*>(p->stage_val[0]), p->task_off + t0, p->chunk_nnz_off, p->chunk_base, n, p->tile_meta, c_col,
      c_val, c_capacity, p->err, nullptr, nullptr, nullptr, 0);
  p->stats.launches += 1;
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}

// Arrays of C with room for `entries`; both or none.
template <typename V>
static bool alloc_c(i64 entries, int32_t** col, V** val, cudaStream_t st) {
  const size_t n = static_cast<size_t>(std::max<i64>(entries, 1));
  *col = static_cast<int32_t*>(dev_alloc(n * sizeof(int32_t), st));
  *val = *col ? static_cast<V*>(dev_alloc(n * sizeof(V), st)) : nullptr;
  if (*val) return true;
  dev_free(*col, st);
  *col = nullptr;
  return false;
}

template <typename V>
static int execute_t(gm_plan* p, cudaStream_t st, gm_csr* C) {
  const gm_csr& A = p->A;
  const gm_csr& B = p->B;
  const i64 nA = A.n_rows;
  gm_plan_info& info = p->info;
  PhaseTimes& tm = p->times;
  p->stats = gm_exec_stats{};
  tm.reset();
  if (p->sink) p->sink->copied = 0;
  cudaEvent_t ev_total0 = nullptr, ev_total1 = nullptr;
  if (tm.enabled) { ev_total0 = tm.get(); ev_total1 = tm.get(); cudaEventRecord(ev_total0, st); }

  HostSlot* const slot = p->slot;
  slot->err[0] = 0;  // (nothing of this plan is in flight: every return of an execute has waited for its streams)
  slot->c_total = 0;
  if (p->row_sums && p->sums_dirty) {
    GM_CUDA(cudaMemsetAsync(p->sums[0], 0, 2 * row_sum_words(nA) * sizeof(u32), st));
  }
  p->sums_dirty = true;  // until the call is through

  // ---- result row_ptr
  i64* c_row_ptr = static_cast<i64*>(dev_alloc(static_cast<size_t>(nA + 1) * sizeof(i64), st));
  int32_t* c_col = nullptr;
  V* c_val = nullptr;
  // ---- light and heavy rows are independent until C.row_ptr is formed: the light rows' kernels go to a second
  // stream, forked from and joined back into the caller's with events (never when single_stream is set)
  bool fork = !p->opts.single_stream && info.rows_heavy > 0 && (info.rows_light > 0 || p->use_tasks);
  SideStream side;
  if (fork) {
    side.st = take_stream();
    if (!side.st || (!p->ev_fork && cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming) != cudaSuccess) ||
        (!p->ev_light && cudaEventCreateWithFlags(&p->ev_light, cudaEventDisableTiming) != cudaSuccess)) {
      cudaGetLastError();
      fork = false;
    }
  }
  cudaStream_t lst = fork ? side.st : st;
  auto fork_light = [&]() { if (fork) { cudaEventRecord(p->ev_fork, st); cudaStreamWaitEvent(lst, p->ev_fork, 0); } };
  auto join_light = [&]() { if (fork) { cudaEventRecord(p->ev_light, lst); cudaStreamWaitEvent(st, p->ev_light, 0); } };
  auto cleanup = [&]() {  // waits for all that is queued: the caller may free or reuse what it reads and writes
    cudaStreamSynchronize(st);
    if (fork) cudaStreamSynchronize(lst);
    if (p->sink && p->sink->copy_stream) cudaStreamSynchronize(p->sink->copy_stream);  // copies out of C in flight
    dev_free(c_row_ptr, st);
    dev_free(c_col, st);
    dev_free(c_val, st);
  };
#define GM_TRY_C(expr) do { int rc2_ = (expr); if (rc2_ != GM_OK) { cleanup(); return rc2_; } } while (0)

  if (!c_row_ptr) { cleanup(); return fail(GM_ERR_OOM, "allocation of C.row_ptr failed"); }
  if (info.rows_heavy > 0) {
    char* const end = p->use_tasks ? reinterpret_cast<char*>(p->task_tickets + 4 * p->batches.size()) : reinterpret_cast<char*>(p->c_total + 16);
    if (cudaMemsetAsync(p->c_total, 0, end - reinterpret_cast<char*>(p->c_total), st) != cudaSuccess) {
      cleanup();
      return fail(GM_ERR_CUDA, std::string("clearing the counters failed: ") + cudaGetErrorString(cudaGetLastError()));
    }
  }

  if (p->use_tasks && p->opts.validate_inputs) GM_TRY_C(validate_tasks<V>(p, st));

  // ---- light rows, all that does not need C (Algorithm 3: Symbolic(A[x_light,:], B), and for most rows the sums too)
  fork_light();
  if (p->use_tasks) GM_TRY_C((task_batch_sums<V, true>(p, 0, st)));  // the longest tasks first
  tm.begin(PhaseTimes::kLightSym, lst);
  GM_TRY_C(light_front<V>(p, lst));
  tm.end(lst);
  if (p->use_tasks) GM_TRY_C((task_batch_sums<V, false>(p, 0, lst)));
  bool light_counted = !fork;  // the heavy path joins before the first prefix sum over the per-row counts
  auto light_rows_to_c = [&](i64 cap, i64 r0, i64 r1, cudaStream_t s2) -> int {
    tm.begin(PhaseTimes::kLightNum, s2);
    const int rc = light_back<V>(p, r0, r1, c_row_ptr, c_col, c_val, cap, s2);
    tm.end(s2);
    return rc;
  };

  const size_t n_batches = p->batches.size();
  i64 capacity = 0;
  i64 total = 0;
  int dev_err = 0;
  bool finished = false;  // small products: counts, C.row_ptr and the totals came from one launch
  if (n_batches <= 1) {
    // ---- everything is resident at once: count, allocate C, then fill
    HeavyBatchState<V> hs;
    if (n_batches == 1 && !p->use_tasks) GM_TRY_C(heavy_batch_front<V>(p, p->batches[0], &hs, st));
    join_light();
    light_counted = true;
    finished = p->finish;
    if (p->use_tasks && !finished) GM_TRY_C(task_batch_counts(p, 0, st));
    tm.begin(PhaseTimes::kScan, st);
    if (finished) {
      k_finish_small<<<1, kFinishThreads, 0, st>>>(p->chunk_nnz, p->task_begin[1], p->chunk_nnz_off, p->row_task_off, info.rows_heavy, p->x_heavy,
                                                   p->row_nnz, nA, c_row_ptr, &slot->c_total, p->chunk_base, kGatherTile, p->tile_meta,
                                                   p->c_total, slot->tail);
      p->stats.launches += 1;
      p->stats.final_chunks += info.rows_heavy * info.params.chunks_required;
      p->stats.staged_products += info.products_heavy;
    } else if (!p->row_sums) {
      p->stats.launches += exclusive_scan<int32_t, i64>(p->row_nnz, c_row_ptr, nA, p->scan_tmp, nullptr, nullptr, nullptr, st,
                                                        reinterpret_cast<i64*>(&slot->c_total));
    }
    tm.end(st);
    if (info.c_nnz_upper * static_cast<i64>(4 + sizeof(V)) <= kCRoomBytes && alloc_c(info.c_nnz_upper, &c_col, &c_val, st)) {
      capacity = info.c_nnz_upper;
    } else {
      if (p->row_sums) {
        k3_total<<<1, 256, 0, st>>>(row_sums_of(p), nA, reinterpret_cast<i64*>(&slot->c_total));
        p->stats.launches += 1;
      }
      if (cudaStreamSynchronize(st) != cudaSuccess) {
        cleanup();
        return fail(GM_ERR_CUDA, std::string("symbolic phase failed: ") + cudaGetErrorString(cudaGetLastError()));
      }
      capacity = total = *static_cast<volatile i64*>(&slot->c_total);
      alloc_c(capacity, &c_col, &c_val, st);
    }
    if (!c_col || !c_val) { cleanup(); return fail(GM_ERR_OOM, "allocation of C (" + std::to_string(capacity) + " entries) failed"); }
    // the heavy and the light rows write different rows of C
    fork_light();
    if (n_batches == 1) {
      tm.begin(PhaseTimes::kAccSym, st);
      if (p->use_tasks) GM_TRY_C(task_batch_gather<V>(p, 0, !finished, c_row_ptr, c_col, c_val, capacity, st));
      else GM_TRY_C((launch_gather<V>(p, p->batches[0], hs, c_row_ptr, c_col, c_val, capacity, st)));
      tm.end(st);
    }
    GM_TRY_C(light_rows_to_c(capacity, 0, nA, lst));
    join_light();
  } else {
    // ---- heavy rows in several staging-buffer fills: C is appended in row order into reserved room
    // Room for C.  Given: use it.  Derived: the structural upper bound sum_i min(IP_i, C.m), cut
    // down to what the device can hold; if the allocator refuses (its own cache can hide free
    // memory from cudaMemGetInfo, or the estimate was too bold) retry with less.
    std::vector<i64> tries;
    if (p->opts.c_capacity > 0) {
      tries.push_back(p->opts.c_capacity);
    } else {
      DeviceFacts facts;
      GM_TRY_C(device_facts(&facts));
      const i64 entry = static_cast<i64>(4 + sizeof(V));
      const i64 inputs = (A.nnz + (&A == &B ? 0 : B.nnz)) * entry + (A.n_rows + B.n_rows + 2) * 8;
      const i64 by_total = (static_cast<i64>(facts.total_mem) - info.workspace_bytes - inputs - (nA + 1) * 8 - (i64{3} << 30)) / entry;
      tries.push_back(std::max<i64>(1, std::min<i64>(info.c_nnz_upper, by_total)));
    }
    for (size_t k = 0; k < tries.size(); ++k) {
      capacity = tries[k];
      if (alloc_c(capacity, &c_col, &c_val, st)) break;
      if (k == 0 && p->opts.c_capacity <= 0) {
        // refused: go down in eight steps to what the device says is free
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) { cudaGetLastError(); break; }
        const i64 by_free = (static_cast<i64>(free_b) - (nA + 1) * 8 - (i64{1} << 30)) / static_cast<i64>(4 + sizeof(V));
        const i64 hi = std::max(capacity, std::min<i64>(info.c_nnz_upper, by_free));
        const i64 lo = std::max<i64>(1, std::min<i64>(info.c_nnz_upper, by_free));
        for (int q = 1; q <= 8 && hi > lo; ++q) tries.push_back(hi - (hi - lo) * q / 8);
      }
    }
    if (!c_col || !c_val) { cleanup(); return fail(GM_ERR_OOM, "allocation of C (room for " + std::to_string(capacity) + " entries) failed"); }
    for (size_t bi = 0; bi < n_batches; ++bi) {
      const Batch& b = p->batches[bi];
      HeavyBatchState<V> hs;
      if (p->use_tasks) {
        if (bi > 0) {  // (the first batch's are already on their way)
          fork_light();
          GM_TRY_C((task_batch_sums<V, true>(p, bi, st)));
          GM_TRY_C((task_batch_sums<V, false>(p, bi, lst)));
        }
        join_light();
        light_counted = true;
        GM_TRY_C(task_batch_counts(p, bi, st));
      } else {
        GM_TRY_C(heavy_batch_front<V>(p, b, &hs, st));
      }
      if (!light_counted) { join_light(); light_counted = true; }
      // rows [r0, r1) of C get their offsets now: every light row in the range was counted up front
      const i64 r0 = bi == 0 ? 0 : p->x_heavy_host[static_cast<size_t>(b.h0)];
      const i64 r1 = bi + 1 == n_batches ? nA : p->x_heavy_host[static_cast<size_t>(p->batches[bi + 1].h0)];
      tm.begin(PhaseTimes::kScan, st);
      p->stats.launches += exclusive_scan<int32_t, i64>(p->row_nnz + r0, c_row_ptr + r0, r1 - r0, p->scan_tmp, p->c_total,
                                                        p->c_total, nullptr, st);
      tm.end(st);
      tm.begin(PhaseTimes::kAccSym, st);
      if (p->use_tasks) GM_TRY_C(task_batch_gather<V>(p, bi, true, c_row_ptr, c_col, c_val, capacity, st));
      else GM_TRY_C((launch_gather<V>(p, b, hs, c_row_ptr, c_col, c_val, capacity, st)));
      tm.end(st);
      if (HostSink* sk = p->sink) {
        // The caller wants C on the host: finish rows [r0, r1) now (their light rows too), note how many entries
        // of C that makes, and send the previous batch's entries on their way while this batch computes.
        GM_TRY_C(light_rows_to_c(capacity, r0, r1, st));
        if (sk->events.size() <= bi) {
          cudaEvent_t ev = nullptr;
          if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) { cleanup(); return fail(GM_ERR_CUDA, "event creation failed"); }
          sk->events.push_back(ev);
        }
        cudaMemcpyAsync(&sk->h_totals[bi], p->c_total, sizeof(i64), cudaMemcpyDeviceToHost, st);
        cudaEventRecord(sk->events[bi], st);
        auto send = [&](size_t done) {
          if (cudaEventSynchronize(sk->events[done]) != cudaSuccess) return;
          const i64 end = std::min<i64>(sk->h_totals[done], sk->capacity);
          if (end > sk->copied) {
            cudaStreamWaitEvent(sk->copy_stream, sk->events[done], 0);
            cudaMemcpyAsync(sk->h_col + sk->copied, c_col + sk->copied, static_cast<size_t>(end - sk->copied) * sizeof(int32_t),
                            cudaMemcpyDeviceToHost, sk->copy_stream);
            cudaMemcpyAsync(static_cast<V*>(sk->h_val) + sk->copied, c_val + sk->copied,
                            static_cast<size_t>(end - sk->copied) * sizeof(V), cudaMemcpyDeviceToHost, sk->copy_stream);
            sk->copied = end;
          }
        };
        if (bi > 0) send(bi - 1);
        if (bi + 1 == n_batches) send(bi);
      }
    }
    if (!p->sink) GM_TRY_C(light_rows_to_c(capacity, 0, nA, st));
  }
  if (tm.enabled) cudaEventRecord(ev_total1, st);
  // [0] nnz(C) so far (several batches), [1] heavy entries; products and entries of small chunks; of mid-size chunks;
  // products and chunks that left the hierarchy early; products the multisplit levels left in place
  if (n_batches > 0 && !finished) cudaMemcpyAsync(slot->tail, p->c_total, kTailWords * sizeof(i64), cudaMemcpyDeviceToHost, st);
  const cudaError_t e2 = cudaStreamSynchronize(st);
  if (e2 != cudaSuccess) {
    cleanup();
    return fail(GM_ERR_CUDA, std::string("execute failed: ") + cudaGetErrorString(e2));
  }
  total = n_batches > 1 ? slot->tail[0] : *static_cast<volatile i64*>(&slot->c_total);
  dev_err = *static_cast<volatile int*>(&slot->err[0]);
  if (dev_err != kDevOk || total > capacity) {
    cleanup();
    if (dev_err == kDevOk) dev_err = kDevCapacity;
    return dev_error_to_status(dev_err);
  }
#undef GM_TRY_C
  if (const i64 entry = static_cast<i64>(4 + sizeof(V));
      n_batches <= 1 && !p->c_is_passing && (capacity - total) * entry > std::max(kCSpareBytes, total * entry)) {
    int32_t* col = nullptr;
    V* val = nullptr;
    if (alloc_c(total, &col, &val, st)) {
      cudaMemcpyAsync(col, c_col, static_cast<size_t>(total) * sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
      cudaMemcpyAsync(val, c_val, static_cast<size_t>(total) * sizeof(V), cudaMemcpyDeviceToDevice, st);
      const cudaError_t e3 = cudaStreamSynchronize(st);
      dev_free(c_col, st);
      dev_free(c_val, st);
      c_col = col;
      c_val = val;
      capacity = total;
      if (e3 != cudaSuccess) {
        cleanup();
        return fail(GM_ERR_CUDA, std::string("moving C failed: ") + cudaGetErrorString(e3));
      }
    }
  }
  p->stats.c_nnz = total;
  if (n_batches > 0) {
    const i64* t = slot->tail;
    p->stats.c_nnz_heavy = t[1];
    p->stats.small_chunk_products = t[2];
    p->stats.small_chunk_entries = t[3];
    p->stats.mid_chunk_products = t[4];
    p->stats.mid_chunk_entries = t[5];
    p->stats.early_exit_products = t[6];
    p->stats.early_exit_chunks = t[7];
    p->stats.split_products -= t[8];
    p->stats.panel_rows = static_cast<float>(t[9]);
    if (p->use_panels && t[9] == 0) drop_panels(p, st);
  }
  p->stats.c_capacity = capacity;
  if (tm.enabled) {
    float ph[PhaseTimes::kCount];
    tm.collect(ph);
    p->stats.ms_light_symbolic = ph[PhaseTimes::kLightSym];
    p->stats.ms_light_numeric = ph[PhaseTimes::kLightNum];
    p->stats.ms_expand = ph[PhaseTimes::kExpand];
    p->stats.ms_histogram = ph[PhaseTimes::kHist];
    p->stats.ms_multisplit = ph[PhaseTimes::kSplit];
    p->stats.ms_gather = ph[PhaseTimes::kAccSym];
    p->stats.ms_accumulate = ph[PhaseTimes::kAccNum];
    p->stats.ms_small_chunks = ph[PhaseTimes::kAccSmall];
    p->stats.ms_mid_chunks = ph[PhaseTimes::kAccMid];
    p->stats.ms_scan = ph[PhaseTimes::kScan];
    cudaEventElapsedTime(&p->stats.ms_total, ev_total0, ev_total1);
  }
  p->sums_at ^= 1;
  p->sums_dirty = false;
  C->n_rows = nA;
  C->n_cols = B.n_cols;
  C->nnz = total;
  C->row_ptr = c_row_ptr;
  C->col_idx = c_col;
  C->vals = c_val;
  C->dtype = A.dtype;
  C->reserved = 0;
  return GM_OK;
}

}  // namespace gm

// ------------------------------------------------------------------------------------------------
// extern "C"
// ------------------------------------------------------------------------------------------------
using namespace gm;

extern "C" {

int gm_set_allocator(gm_alloc_fn alloc_fn, gm_free_fn free_fn, void* user) {
  if ((alloc_fn == nullptr) != (free_fn == nullptr)) return fail(GM_ERR_INVALID_ARG, "alloc and free must be given together");
  g_alloc.alloc = alloc_fn;
  g_alloc.free = free_fn;
  g_alloc.user = user;
  return GM_OK;
}

int gm_spgemm_plan_ex(const gm_csr* A, const gm_csr* B, size_t smem_bytes, const gm_plan_opts* opts, void* cuda_stream,
                      gm_plan** plan_out) {
  if (!plan_out) return fail(GM_ERR_INVALID_ARG, "plan_out is null");
  *plan_out = nullptr;
  GM_TRY(check_csr_arg(A, "A"));
  GM_TRY(check_csr_arg(B, "B"));
  if (A->dtype != B->dtype) return fail(GM_ERR_DTYPE, "A and B have different value types");
  if (A->n_cols != B->n_rows) return fail(GM_ERR_DIM_MISMATCH, "A.n_cols != B.n_rows");
  gm_plan* p = new gm_plan();
  p->A = *A;
  p->B = *B;
  p->sv = value_bytes(A->dtype);
  p->smem_bytes = smem_bytes;
  if (opts) p->opts = *opts;
  p->plan_stream = static_cast<cudaStream_t>(cuda_stream);
  const char* env = std::getenv("GM_TIMING");
  p->times.enabled = env && env[0] == '1';
  const int rc = build_plan(p, p->plan_stream);
  if (rc != GM_OK) {
    cudaStreamSynchronize(p->plan_stream);
    gm_plan_destroy(p);
    return rc;
  }
  if (p->pending && (cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
                     cudaStreamGetId(p->plan_stream, &p->plan_stream_id) != cudaSuccess ||
                     cudaEventRecord(p->ev_fork, p->plan_stream) != cudaSuccess)) {
    cudaStreamSynchronize(p->plan_stream);
    gm_plan_destroy(p);
    return fail(GM_ERR_CUDA, std::string("end of planning: ") + cudaGetErrorString(cudaGetLastError()));
  }
  *plan_out = p;
  return GM_OK;
}

int gm_spgemm_plan(const gm_csr* A, const gm_csr* B, size_t smem_bytes, gm_plan** plan_out) {
  return gm_spgemm_plan_ex(A, B, smem_bytes, nullptr, nullptr, plan_out);
}

int gm_spgemm_execute(gm_plan* plan, void* cuda_stream, gm_csr* C_out) {
  if (!plan || !C_out) return fail(GM_ERR_INVALID_ARG, "plan or C_out is null");
  std::memset(C_out, 0, sizeof(*C_out));
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (plan->pending) {
    unsigned long long id = 0;
    GM_CUDA(cudaStreamGetId(st, &id));
    if (id != plan->plan_stream_id) GM_CUDA(cudaStreamWaitEvent(st, plan->ev_fork, 0));
  }
  auto run = [&]() { return plan->A.dtype == GM_F32 ? execute_t<float>(plan, st, C_out) : execute_t<double>(plan, st, C_out); };
  if (plan->light_relist) GM_TRY(light_rows_by_hash(plan, st));  // (an execute before this one had no room for the lists)
  if (plan->task_replan) GM_TRY(tasks_without_panels(plan, st));
  int rc = run();
  plan->pending = false;  // (whatever the result, the execute has waited for its stream)
  auto no_room = [&]() { return rc == GM_ERR_OOM || (rc == GM_ERR_CAPACITY && plan->opts.c_capacity <= 0); };
  if (plan->use_panels && no_room()) {  // C does not fit beside the panels' lists: once more without them
    GM_TRY(tasks_without_panels(plan, st));
    rc = run();
  }
  if (plan->light_stage && no_room()) {  // ... nor beside the light rows' staging area
    GM_TRY(light_rows_by_hash(plan, st));
    rc = run();
  }
  return rc;
}

int gm_plan_get_info(const gm_plan* plan, gm_plan_info* out) {
  if (!plan || !out) return fail(GM_ERR_INVALID_ARG, "null argument");
  *out = plan->info;
  return GM_OK;
}

int gm_exec_get_stats(const gm_plan* plan, gm_exec_stats* out) {
  if (!plan || !out) return fail(GM_ERR_INVALID_ARG, "null argument");
  *out = plan->stats;
  return GM_OK;
}

int gm_plan_set_timing(gm_plan* plan, int enable) {
  if (!plan) return fail(GM_ERR_INVALID_ARG, "null plan");
  plan->times.enabled = enable != 0;
  return GM_OK;
}

int gm_plan_get_row_products(const gm_plan* plan, int64_t* ip_out_device, void* cuda_stream) {
  if (!plan || !ip_out_device) return fail(GM_ERR_INVALID_ARG, "null argument");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (plan->A.n_rows > 0)
    GM_CUDA(cudaMemcpyAsync(ip_out_device, plan->ip, static_cast<size_t>(plan->A.n_rows) * sizeof(int64_t),
                            cudaMemcpyDeviceToDevice, st));
  return GM_OK;
}

void gm_csr_free(gm_csr* C) {
  if (!C) return;
  dev_free(const_cast<int64_t*>(C->row_ptr), nullptr);
  dev_free(const_cast<int32_t*>(C->col_idx), nullptr);
  dev_free(const_cast<void*>(C->vals), nullptr);
  std::memset(C, 0, sizeof(*C));
}

void gm_plan_destroy(gm_plan* plan) {
  if (!plan) return;
  if (plan->pending && plan->ev_fork) cudaEventSynchronize(plan->ev_fork);
  if (plan->ev_fork) cudaEventDestroy(plan->ev_fork);
  if (plan->ev_light) cudaEventDestroy(plan->ev_light);
  for (auto& b : plan->owned) dev_free(b.p, plan->plan_stream);
  give_slot(plan->slot);
  delete plan;
}

int gm_spgemm_host(const gm_csr* A_host, const gm_csr* B_host, size_t smem_bytes, const gm_plan_opts* opts, gm_csr* C_host,
                   int64_t c_capacity) {
  GM_TRY(check_csr_arg(A_host, "A_host"));
  GM_TRY(check_csr_arg(B_host, "B_host"));
  if (!C_host || !C_host->row_ptr || c_capacity < 0) return fail(GM_ERR_INVALID_ARG, "C_host needs caller-owned buffers");
  if (A_host->dtype != B_host->dtype) return fail(GM_ERR_DTYPE, "A and B have different value types");
  const size_t sv = static_cast<size_t>(value_bytes(A_host->dtype));
  cudaStream_t st = take_stream();
  if (!st) return fail(GM_ERR_CUDA, "stream creation failed");
  gm_csr dev[2];
  std::vector<void*> tmp;
  int rc = GM_OK;
  auto upload = [&](const gm_csr* H, gm_csr* D) -> int {
    *D = *H;
    const size_t rp_bytes = (static_cast<size_t>(H->n_rows + 1) * 8 + 255) & ~size_t{255};
    const size_t ci_bytes = (static_cast<size_t>(H->nnz) * 4 + 255) & ~size_t{255};
    char* rp = static_cast<char*>(dev_alloc(rp_bytes + ci_bytes + static_cast<size_t>(H->nnz) * sv, st));
    if (!rp) return fail(GM_ERR_OOM, "device allocation for an input failed");
    tmp.push_back(rp);
    char* ci = rp + rp_bytes;
    char* va = ci + ci_bytes;
    GM_CUDA(cudaMemcpyAsync(rp, H->row_ptr, static_cast<size_t>(H->n_rows + 1) * 8, cudaMemcpyHostToDevice, st));
    if (H->nnz > 0) {
      GM_CUDA(cudaMemcpyAsync(ci, H->col_idx, static_cast<size_t>(H->nnz) * 4, cudaMemcpyHostToDevice, st));
      GM_CUDA(cudaMemcpyAsync(va, H->vals, static_cast<size_t>(H->nnz) * sv, cudaMemcpyHostToDevice, st));
    }
    D->row_ptr = reinterpret_cast<const int64_t*>(rp);
    D->col_idx = reinterpret_cast<const int32_t*>(ci);
    D->vals = va;
    return GM_OK;
  };
  gm_plan* plan = nullptr;
  gm_csr C{};
  rc = upload(A_host, &dev[0]);
  // a matrix multiplied with itself is sent once
  const bool same = A_host->n_rows == B_host->n_rows && A_host->n_cols == B_host->n_cols && A_host->nnz == B_host->nnz &&
                    A_host->row_ptr == B_host->row_ptr && A_host->col_idx == B_host->col_idx && A_host->vals == B_host->vals;
  if (rc == GM_OK && same) dev[1] = dev[0];
  else if (rc == GM_OK) rc = upload(B_host, &dev[1]);
  if (rc == GM_OK) rc = gm_spgemm_plan_ex(&dev[0], &dev[1], smem_bytes, opts, st, &plan);
  // With several batches, C's entries travel to the host batch by batch while later batches compute.
  HostSink sink;
  bool use_sink = false;
  if (rc == GM_OK && plan->batches.size() > 1 && C_host->col_idx && C_host->vals && c_capacity > 0) {
    sink.h_col = const_cast<int32_t*>(C_host->col_idx);
    sink.h_val = const_cast<void*>(C_host->vals);
    sink.capacity = c_capacity;
    use_sink = cudaStreamCreateWithFlags(&sink.copy_stream, cudaStreamNonBlocking) == cudaSuccess &&
               cudaMallocHost(reinterpret_cast<void**>(&sink.h_totals), plan->batches.size() * sizeof(int64_t)) == cudaSuccess;
    if (use_sink) plan->sink = &sink;
  }
  if (plan) plan->c_is_passing = true;
  if (rc == GM_OK) rc = gm_spgemm_execute(plan, st, &C);
  if (plan) plan->sink = nullptr;
  if (rc == GM_OK) {
    C_host->n_rows = C.n_rows;
    C_host->n_cols = C.n_cols;
    C_host->nnz = C.nnz;
    C_host->dtype = C.dtype;
    cudaError_t e = cudaMemcpyAsync(const_cast<int64_t*>(C_host->row_ptr), C.row_ptr, static_cast<size_t>(C.n_rows + 1) * 8,
                                    cudaMemcpyDeviceToHost, st);
    if (C.nnz > c_capacity) {
      rc = fail(GM_ERR_CAPACITY, "C has " + std::to_string(C.nnz) + " entries, more than c_capacity");
    } else if (C.nnz > 0 && e == cudaSuccess) {
      if (!C_host->col_idx || !C_host->vals) {
        rc = fail(GM_ERR_INVALID_ARG, "C_host->col_idx / vals are null");
      } else {
        const int64_t done = use_sink ? sink.copied : 0;  // entries the batches have already sent
        if (C.nnz > done) {
          e = cudaMemcpyAsync(const_cast<int32_t*>(C_host->col_idx) + done, C.col_idx + done,
                              static_cast<size_t>(C.nnz - done) * 4, cudaMemcpyDeviceToHost, st);
          if (e == cudaSuccess)
            e = cudaMemcpyAsync(static_cast<char*>(const_cast<void*>(C_host->vals)) + static_cast<size_t>(done) * sv,
                                static_cast<const char*>(C.vals) + static_cast<size_t>(done) * sv,
                                static_cast<size_t>(C.nnz - done) * sv, cudaMemcpyDeviceToHost, st);
        }
      }
    }
    if (use_sink && cudaStreamSynchronize(sink.copy_stream) != cudaSuccess && e == cudaSuccess) e = cudaErrorUnknown;
    cudaError_t e2 = cudaStreamSynchronize(st);
    if (rc == GM_OK && (e != cudaSuccess || e2 != cudaSuccess)) rc = fail(GM_ERR_CUDA, "copy of C to the host failed");
    dev_free(const_cast<int64_t*>(C.row_ptr), st);
    dev_free(const_cast<int32_t*>(C.col_idx), st);
    dev_free(const_cast<void*>(C.vals), st);
  }
  if (plan) {
    plan->plan_stream = st;
    gm_plan_destroy(plan);
  }
  for (void* q : tmp) dev_free(q, st);
  cudaStreamSynchronize(st);
  if (sink.copy_stream) {
    cudaStreamSynchronize(sink.copy_stream);
    cudaStreamDestroy(sink.copy_stream);
  }
  for (cudaEvent_t ev : sink.events) cudaEventDestroy(ev);
  if (sink.h_totals) cudaFreeHost(sink.h_totals);
  give_stream(st);
  return rc;
}

const char* gm_status_string(int status) {
  switch (status) {
    case GM_OK: return "GM_OK";
    case GM_ERR_INVALID_ARG: return "GM_ERR_INVALID_ARG";
    case GM_ERR_DIM_MISMATCH: return "GM_ERR_DIM_MISMATCH";
    case GM_ERR_DTYPE: return "GM_ERR_DTYPE";
    case GM_ERR_BAD_CSR: return "GM_ERR_BAD_CSR";
    case GM_ERR_OOM: return "GM_ERR_OOM";
    case GM_ERR_CAPACITY: return "GM_ERR_CAPACITY";
    case GM_ERR_CUDA: return "GM_ERR_CUDA";
    case GM_ERR_TIMEOUT: return "GM_ERR_TIMEOUT";
    case GM_ERR_UNSUPPORTED_SMEM: return "GM_ERR_UNSUPPORTED_SMEM";
    case GM_ERR_INTERNAL: return "GM_ERR_INTERNAL";
    default: return "GM_ERR_UNKNOWN";
  }
}

const char* gm_last_error(void) { return g_last_error.c_str(); }

}  // extern "C"

// ------------------------------------------------------------------------------------------------
// Row analysis without any allocation (see gm_row_products_noalloc in gmagnus.h)
// ------------------------------------------------------------------------------------------------
namespace gm {

constexpr i64 kNoAllocMaxNnz = GM_NOALLOC_MAX_NNZ_A;

}  // namespace gm

extern "C" int gm_row_products_noalloc(const gm_csr* A, const gm_csr* B, int64_t* ip_out_device, void* cuda_stream) {
  GM_TRY(check_csr_arg(A, "A", true));
  GM_TRY(check_csr_arg(B, "B", true));
  if (!ip_out_device && A->n_rows > 0) return fail(GM_ERR_INVALID_ARG, "ip_out_device is null");
  if (A->n_cols != B->n_rows) return fail(GM_ERR_DIM_MISMATCH, "A.n_cols != B.n_rows");
  if (A->nnz > kNoAllocMaxNnz)
    return fail(GM_ERR_CAPACITY, "gm_row_products_noalloc handles at most " + std::to_string(kNoAllocMaxNnz) +
                                     " stored entries of A (got " + std::to_string(A->nnz) + ")");
  DeviceFacts facts;
  GM_TRY(device_facts(&facts));
  if (A->n_rows == 0) return GM_OK;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int T = k1_tile_items(A->n_rows, A->nnz, facts.num_sms);
  const unsigned grid = static_cast<unsigned>((A->n_rows + A->nnz + T - 1) / T);
  const bool wide = B->n_cols > (i64{1} << 24);
  auto kern = T == kK1Small ? (wide ? k1_row_products_only<kK1Small, i64> : k1_row_products_only<kK1Small, u32>)
                            : (wide ? k1_row_products_only<kK1Large, i64> : k1_row_products_only<kK1Large, u32>);
  GM_CUDA(cudaMemsetAsync(ip_out_device, 0, static_cast<size_t>(A->n_rows) * sizeof(int64_t), st));
  kern<<<grid, kK1Threads, 0, st>>>(A->row_ptr, A->col_idx, A->n_rows, A->nnz, B->row_ptr, ip_out_device);
  GM_CUDA(cudaGetLastError());
  return GM_OK;
}
