// Internal declarations shared by the translation units of libhnv.so.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <utility>
#include <vector>

#include "hnv.h"

namespace hnv {

// ---------------------------------------------------------------------------
// Errors
// ---------------------------------------------------------------------------

// Records a one-line message for hnv_last_error_detail() (thread-local).
void set_error_detail(const char* fmt, ...);
void clear_error_detail();
int cuda_status(cudaError_t e, const char* what);

#define HNV_FAIL(code, ...)                 \
  do {                                      \
    ::hnv::set_error_detail(__VA_ARGS__);   \
    return (code);                          \
  } while (0)

#define HNV_CHECK(expr)                     \
  do {                                      \
    int hnv_s_ = (expr);                    \
    if (hnv_s_ != HNV_OK) return hnv_s_;    \
  } while (0)

#define HNV_CUDA(call)                                             \
  do {                                                             \
    cudaError_t hnv_e_ = (call);                                   \
    if (hnv_e_ != cudaSuccess) return ::hnv::cuda_status(hnv_e_, #call); \
  } while (0)

// Bits of the per-graph device error word (set with atomicOr by kernels that
// validate input; read back by the host after a synchronising step).
enum : int32_t {
  ERRBIT_NODE_RANGE = 1,    // an input node ID outside [0, n)
  ERRBIT_EMPTY_EDGE = 2,    // an input hyperedge with no members
  ERRBIT_BAD_WEIGHT = 4,    // a weight that is not finite and > 0
  ERRBIT_BAD_PTR = 8,       // edge_ptr not starting at 0 / decreasing
  ERRBIT_TIMEOUT = 16,      // a bounded device wait gave up (refinement)
  ERRBIT_BAD_ITEM = 32,     // a batched work item outside its graph's arrays (skipped)
  ERRBIT_BAD_FEATURE = 64   // a node feature that is not finite or exceeds 1e15 in magnitude
};

// ---------------------------------------------------------------------------
// Kernel launches
// ---------------------------------------------------------------------------

void note_launch();
void note_launches(int64_t k);   // k kernels at once (a replayed CUDA graph)
int num_sms();   // of the current device

// Launches kernel<<<grid, block, smem, s>>>(args...) and counts it. A launch
// with no blocks is skipped.
template <typename... KArgs, typename... Args>
int launch(const char* name, void (*kernel)(KArgs...), unsigned grid, unsigned block,
           size_t smem, cudaStream_t s, Args&&... args) {
  if (grid == 0) return HNV_OK;
  kernel<<<grid, block, smem, s>>>(static_cast<KArgs>(std::forward<Args>(args))...);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, name);
  return HNV_OK;
}

// Blocks for a grid-stride loop over `items` with `per_block` items per
// block, capped at `waves` blocks per SM.
unsigned grid_for(int64_t items, int64_t per_block, int waves = 8);

// ---------------------------------------------------------------------------
// Device memory (stream-ordered; replaceable through hnv_set_allocator)
// ---------------------------------------------------------------------------

int dev_alloc(void** p, size_t bytes, cudaStream_t s);
void dev_free(void* p, cudaStream_t s);

// Temporary device buffers released (stream-ordered) when the pool dies.
// Small ones are cut from slabs: a level of a 2,000-node graph asks for about
// 25 of them, and each allocation with its release costs the host 2-3 us. Where
// a slab cannot be had (an allocator hook with little memory), each is
// allocated by itself.
class TempPool {
 public:
  explicit TempPool(cudaStream_t s) : s_(s) {}
  ~TempPool() {
    for (void* p : ptrs_) dev_free(p, s_);
  }
  TempPool(const TempPool&) = delete;
  TempPool& operator=(const TempPool&) = delete;
  template <typename T>
  int get(T** out, size_t count) {
    const size_t bytes = ((count ? count : 1) * sizeof(T) + 255) & ~(size_t)255;
    void* p = nullptr;
    if (bytes <= kSlab / 4 && !no_slabs_) {
      if (left_ < bytes) {
        if (dev_alloc(&p, kSlab, s_) == HNV_OK) {
          ptrs_.push_back(p);
          at_ = static_cast<char*>(p);
          left_ = kSlab;
        } else {
          clear_error_detail();
          no_slabs_ = true;
        }
      }
      if (!no_slabs_) {
        *out = reinterpret_cast<T*>(at_);
        at_ += bytes;
        left_ -= bytes;
        return HNV_OK;
      }
    }
    HNV_CHECK(dev_alloc(&p, bytes, s_));
    ptrs_.push_back(p);
    *out = static_cast<T*>(p);
    return HNV_OK;
  }

 private:
  static constexpr size_t kSlab = 512 * 1024;
  cudaStream_t s_;
  char* at_ = nullptr;
  size_t left_ = 0;
  bool no_slabs_ = false;
  std::vector<void*> ptrs_;
};

// ---------------------------------------------------------------------------
// Phase timing (CUDA events on the launching stream)
// ---------------------------------------------------------------------------

bool timing_on();
// Records the start event of a phase; returns an opaque slot or -1.
int timing_begin(int phase, cudaStream_t s, double alg_bytes);
void timing_end(int slot, cudaStream_t s);

// An NVTX range (named in profiler timelines) for the scope's lifetime.
// NVTX is header-only: without a tool attached a range costs a check.
struct NvtxRange {
  explicit NvtxRange(const char* fmt, ...);
  ~NvtxRange();
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

struct PhaseScope {
  int slot;
  cudaStream_t s;
  PhaseScope(int phase, cudaStream_t st, double bytes) : slot(-1), s(st) {
    if (timing_on()) slot = timing_begin(phase, st, bytes);
  }
  ~PhaseScope() {
    if (slot >= 0) timing_end(slot, s);
  }
};

// ---------------------------------------------------------------------------
// Primitives (prims.cu)
// ---------------------------------------------------------------------------

// out[i] = sum_{j<i} in[i]; in == out allowed. If total != nullptr the sum of
// all n inputs is written to *total (device). n may be 0.
int exclusive_scan_i32(const int32_t* in, int32_t* out, int64_t n, int32_t* total,
                       cudaStream_t s);

// Stable LSD radix sort of 64-bit keys, one pass of 8 bits per entry of
// `shifts` (digit = (key >> shift) & 255), ping-ponging between keys and alt.
// *result receives whichever buffer holds the sorted keys.
int radix_sort_u64(uint64_t* keys, uint64_t* alt, int64_t n, const int* shifts,
                   int npasses, cudaStream_t s, uint64_t** result);

// Shifts for the passes that sort the low `low_bits` bits, then bits
// [32, 32 + high_bits). Returns the number of passes.
int radix_shifts(int low_bits, int high_bits, int* shifts);

// Number of bits needed to hold values in [0, count).
int bits_for_count(int64_t count);

// Last index i in [0, n) with ptr[i] <= key (ptr ascending, ptr[0] <= key),
// found by one warp 32 probes at a time.
template <typename P>
__device__ __forceinline__ int64_t warp_last_le(const P* __restrict__ ptr, int64_t n, int64_t key) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;   // the answer is in [lo, hi)
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t at = lo + lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, at < hi && (int64_t)ptr[at] <= key);
    const int last = 31 - __clz((int)le);   // lane 0 always holds
    const int64_t nlo = lo + last * step;
    hi = nlo + step < hi ? nlo + step : hi;
    lo = nlo;
  }
  return lo;
}

// Visits every entry k of the rows [0, rows) of a CSR with offsets ptr as
// f(row, k): a block of kEntryThreads takes kEntryTile consecutive entries,
// finds the rows they lie in, marks each row's first entry in shared memory
// and spreads the marks by a running maximum. Every thread has the same work
// whatever the row lengths, and accesses by k are coalesced. (Rows dealt to
// warps left one warp on a row of thousands of entries: packing the 17.6M
// incidences of the 1M-node workload took 283 us.) Launch with one block per
// tile of the `total` entries; total = ptr[rows].
constexpr int kEntryThreads = 256;
constexpr int kEntryTile = 2048;
inline unsigned entry_grid(int64_t total) {
  return (unsigned)((total + kEntryTile - 1) / kEntryTile);
}

template <typename P, typename F>
__device__ __forceinline__ void csr_entries_visit(int64_t rows, const P* __restrict__ ptr,
                                                  int64_t total, F f) {
  constexpr int PER = kEntryTile / kEntryThreads;
  __shared__ int32_t mark[kEntryTile];
  __shared__ int32_t wmax[kEntryThreads / 32];
  __shared__ int64_t bounds[2];
  const int64_t t0 = (int64_t)blockIdx.x * kEntryTile;
  const int64_t t1 = t0 + kEntryTile < total ? t0 + kEntryTile : total;
  if (t0 >= t1) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w < 2) {
    const int64_t r = warp_last_le(ptr, rows, w == 0 ? t0 : t1 - 1);
    if (lane == 0) bounds[w] = r;
  }
  for (int i = threadIdx.x; i < kEntryTile; i += kEntryThreads) mark[i] = 0;
  __syncthreads();
  const int64_t r0 = bounds[0], r1 = bounds[1];
  // (an empty row shares its start with the row after it: the larger wins)
  for (int64_t r = r0 + 1 + threadIdx.x; r <= r1; r += kEntryThreads)
    atomicMax(&mark[(int64_t)ptr[r] - t0], (int32_t)(r - r0));
  __syncthreads();
  int32_t x[PER], run = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    run = max(run, mark[threadIdx.x * PER + j]);
    x[j] = run;
  }
  int32_t inc = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc = max(inc, y);
  }
  if (lane == 31) wmax[w] = inc;
  int32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 0) before = 0;
  __syncthreads();
  for (int q = 0; q < w; ++q) before = max(before, wmax[q]);
#pragma unroll
  for (int j = 0; j < PER; ++j) mark[threadIdx.x * PER + j] = max(x[j], before);
  __syncthreads();
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = j * kEntryThreads + threadIdx.x;
    if (t0 + i < t1) f(r0 + mark[i], t0 + i);
  }
}

// Compaction of entries [0, n) chosen by a predicate, in order, without
// materialised flags: compact_count writes the chosen per tile (and marks
// nothing), the tile counts are scanned, compact_write recomputes the
// predicate and calls put(k, position).
constexpr int kCompactThreads = 256;
constexpr int kCompactTile = 4096;
inline int64_t compact_tiles(int64_t n) { return (n + kCompactTile - 1) / kCompactTile; }

template <typename Pred>
__device__ __forceinline__ void compact_count(int64_t n, int32_t* __restrict__ tile_count, Pred pred) {
  const int64_t t0 = (int64_t)blockIdx.x * kCompactTile;
  int32_t c = 0;
#pragma unroll 4
  for (int j = 0; j < kCompactTile / kCompactThreads; ++j) {
    const int64_t k = t0 + j * kCompactThreads + threadIdx.x;
    if (k < n && pred(k)) ++c;
  }
  __shared__ int32_t ws[kCompactThreads / 32];
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < kCompactThreads / 32; ++q) c += ws[q];
    tile_count[blockIdx.x] = c;
  }
}

template <typename Pred, typename Put>
__device__ __forceinline__ void compact_write(int64_t n, const int32_t* __restrict__ tile_off,
                                              Pred pred, Put put) {
  // a warp takes 512 consecutive entries, 32 at a time: ballots rank them
  constexpr int ROUNDS = kCompactTile / kCompactThreads;
  __shared__ int32_t ws[kCompactThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kCompactTile + (int64_t)w * (32 * ROUNDS) + lane;
  unsigned bits[ROUNDS];
  int32_t c = 0;
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const int64_t k = base + j * 32;
    bits[j] = __ballot_sync(0xffffffffu, k < n && pred(k));
    c += __popc(bits[j]);
  }
  if (lane == 0) ws[w] = c;
  __syncthreads();
  int32_t at = tile_off[blockIdx.x];
  for (int q = 0; q < w; ++q) at += ws[q];
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    if (bits[j] >> lane & 1u) put(base + j * 32, at + __popc(bits[j] & ((1u << lane) - 1u)));
    at += __popc(bits[j]);
  }
}

// Sorts keys[ptr[i] .. ptr[i+1]) of every segment i < segs by their low 32
// bits (stable is irrelevant: keys within a segment share their high word).
// ptr is int32 (ptr32) or int64 (ptr64, when ptr32 is null); max_len bounds
// the segment lengths and must be <= kSegSortMax.
// distinct_range > 0 promises that every low word is < distinct_range and
// that the caller needs only each segment's sorted distinct values: segments
// of more than 256 keys then hold their distinct values ascending followed by
// copies of the largest (still sorted; only the multiplicities differ), when
// a bitmap of distinct_range bits fits kSegBitmapBytes of shared memory.
constexpr int32_t kSegSortMax = 8192;
constexpr size_t kSegBitmapBytes = 160 * 1024;
int segmented_sort_low32(int32_t segs, const int32_t* ptr32, const int64_t* ptr64,
                         int32_t max_len, int64_t total_keys, uint64_t* keys, cudaStream_t s,
                         uint32_t distinct_range = 0);

// The distinct keys of n sorted (row << 32 | col) keys as a CSR, in two
// steps: unique_count leaves the kept keys' offsets per tile in tiles
// [compact_tiles(n)] and their number in *total (device); unique_csr writes
// their cols and row_ptr[row] of every row that has keys.
int unique_count(const uint64_t* keys, int64_t n, int32_t* tiles, int32_t* total, cudaStream_t s);
int unique_csr(const uint64_t* keys, int64_t n, const int32_t* tiles, int32_t* cols,
               int32_t* row_ptr, cudaStream_t s);

int fill_i32(int32_t* p, int32_t value, int64_t n, cudaStream_t s);

// CSC (transpose) of a CSR with ascending rows: col_ptr[n_cols+1] and
// col_rows[nnz] with ascending entries per column.
int transpose_csr(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t* row_ptr,
                  const int32_t* cols, int32_t* col_ptr, int32_t* col_rows, cudaStream_t s);

// ---------------------------------------------------------------------------
// The hierarchy
// ---------------------------------------------------------------------------

// Work plan of one half-sweep (one side of the star expansion).
// Rows are put in classes by length: A (1..4 incidences), B (5..16),
// C (17..64), D (65..T); longer rows are cut into chunks of T consecutive
// incidences whose partial sums a second kernel reduces in chunk order.
// `items` holds one descriptor per work item {row, first incidence, length,
// partial slot or -1}: the A rows, then B, C, D, then every chunk. Split
// rows are listed in `long_desc` {row, first chunk, chunk count, 0}: those
// with at most kMidChunks chunks first, then the rest. Rows of length 0 are
// in zero_rows.
constexpr int32_t kSplitT = 128;
constexpr int32_t kMidChunks = 32;

// Class boundaries of a plan (lengths: A <= a_max < B <= b_max < C <= c_max
// < D <= T). The single-graph path uses the defaults; the batched path takes
// them from its autotuner.
struct PlanShape {
  int32_t a_max = 4;
  int32_t b_max = 16;
  int32_t c_max = 64;
};

struct SplitPlan {
  int32_t T = kSplitT;
  int32_t n_a = 0, n_b = 0, n_c = 0, n_d = 0;  // rows per class
  int32_t n_chunks = 0;                        // chunk items (after the D rows)
  int32_t n_mid = 0, n_huge = 0;               // split rows by chunk count
  int32_t n_mid_chunks = 0;                    // chunk items of the n_mid rows (they come first)
  int32_t n_zero = 0;
  int4* items = nullptr;              // [n_a + n_b + n_c + n_d + n_chunks]
  int4* long_desc = nullptr;          // [n_mid + n_huge]
  int32_t* zero_rows = nullptr;       // [n_zero]
  // the neighbours of the class-A rows (at most 4; unused slots 0), one
  // int4 per class-A item in item order, or null (see build_split_plan)
  int4* a_members = nullptr;          // [n_a]
  // the same for the class-B rows (at most 16 neighbours, 16 slots each)
  int32_t* b_members = nullptr;       // [n_b * 16]
};

struct Level {
  int32_t n = 0, m = 0;
  int64_t nnz = 0;
  int32_t* e_ptr = nullptr;      // [m+1]
  int32_t* e_nodes = nullptr;    // [nnz]
  int32_t* v_ptr = nullptr;      // [n+1]
  int32_t* v_edges = nullptr;    // [nnz]
  float* w = nullptr;            // [m]
  float* v_w = nullptr;          // [nnz] w of each CSC entry
  float* deg_v = nullptr;        // [n] sum_{e ∋ v} w_e
  float* inv_deg_v = nullptr;    // [n] 1/deg_v (0 if no hyperedge)
  float* inv_size_e = nullptr;   // [m] 1/|e|
  int32_t* orig_e = nullptr;     // [m] level-0 ID
  int32_t* rep_v = nullptr;      // [n] -> level+1 (null on the coarsest)
  int32_t* rep_e = nullptr;      // [m] -> level+1 or -1-c
  float* feat = nullptr;         // [n x feat_k] node features (cosine policy), or null
  int32_t feat_k = 0;
  SplitPlan planE, planV;
  // adjoint (built on first use; freed with the level)
  bool adj_ready = false;
  float* v_invsize_w = nullptr;  // [nnz] CSC order: 1/|e| of each hyperedge
  int32_t* ch_ptr = nullptr;     // [n_{l+1}+1] children of each coarse node:
  int32_t* ch_idx = nullptr;     //   fine nodes v, then collapsed hyperedges n + e
  int64_t ch_total = 0;          // entries of ch_idx
  SplitPlan planC;
  std::vector<void*> owned;      // every device allocation of this level
  // panel plans of the two sides (0 hyperedge rows, 1 node rows) for the
  // row size they were chosen for (side_plan); kept apart from `owned` so
  // that they can be rebuilt for another row size
  SplitPlan panel_plan[2];
  int32_t panel_P[2] = {1, 1};
  size_t panel_rb[2] = {0, 0};
  std::vector<void*> panel_owned[2];
};

struct TeamLevel;
// Limit of one barrier wait of the team kernel.
constexpr uint64_t kTeamWaitNs = 4000000000ull;
// 32-bit words a one-graph team launch owns: the barrier line, the stopping
// rule's 3 running maxima and its 3 results.
constexpr int kTeamWords = 64, kTeamDelta = 32, kTeamResult = 36;

// Whose launches use a graph's k-th set of these words. Launches on one stream
// follow each other and share a set; launches on other streams may run beside
// them (a graph without split rows shares no other scratch), and so may the
// replays of a capture, whose set is its own for the graph's lifetime. A call
// neither allocates the words nor gives them back.
struct TeamSlot {
  bool taken = false;
  unsigned long long stream = 0;    // cudaStreamGetId (not reused); in a capture the handle
  unsigned long long capture = 0;   // id of the capture, 0: none
  uint64_t used = 0;                // turn of the last launch (none captured)
  cudaEvent_t done = nullptr;       // after it: another stream may take the set
};
constexpr int kTeamSlots = 32, kTeamStreamSlots = 8;   // sets; of them kept for streams
constexpr int kTeamLevels = 40;   // levels a graph has room to describe from the start

}  // namespace hnv

struct hnv_graph {
  int device = 0;
  cudaStream_t stream = nullptr;
  std::vector<hnv::Level> levels;
  int32_t* d_err = nullptr;      // device error word
  int32_t* h_buf = nullptr;      // pinned host scratch (64 ints)
  int32_t* d_buf = nullptr;      // device scratch (64 ints)
  // one allocation: d_err, d_buf, kTeamSlots x kTeamWords team_words and
  // kTeamLevels of the team_levels
  int32_t* d_words = nullptr;
  int32_t* team_words = nullptr;
  hnv::TeamSlot team_slots[hnv::kTeamSlots];
  uint64_t team_turn = 0;
  hnv::TeamLevel* team_buf = nullptr;
  // device, one per level (team.cu): team_buf, or an allocation of its own
  hnv::TeamLevel* team_levels = nullptr;
  // hnv_selftest_team_timeout: of the one-launch calls' barriers
  uint64_t team_wait_ns = hnv::kTeamWaitNs;
  int32_t team_stop_at = 0;
  bool team_refuse = false;      // hnv_selftest_team_refuse
  float* partials = nullptr;     // split-row partial sums
  size_t partials_bytes = 0;
  float* jacobi_tmp = nullptr;   // Jacobi: next hyperedge rows
  size_t jacobi_bytes = 0;
  // a capture uses the scratch above: what is outgrown is kept for its replays
  bool captured = false;
  std::vector<void*> outgrown;
  uint64_t generation = 0;       // bumped whenever the hierarchy is rebuilt
  // side streams on which a half-sweep's row classes run concurrently
  // (forked from and joined back into the caller's stream)
  cudaStream_t aux[2] = {nullptr, nullptr};
  cudaEvent_t fork_ev = nullptr;
  cudaEvent_t join_ev[2] = {nullptr, nullptr};
};

namespace hnv {

// incidence.cu: level-0 construction, derived arrays and split plans.
int build_level0(hnv_graph* g, int32_t n, int32_t m, const int64_t* d_edge_ptr,
                 const int32_t* d_edge_nodes, const float* d_w, Level* out);
int finish_level(hnv_graph* g, Level* lv);   // derived arrays + plans
// Weight-dependent arrays of a level (v_w, deg_v, inv_deg_v) from lv->w.
int level_weight_arrays(Level* lv, cudaStream_t s);
// Split-row work plan of a CSR with `rows` rows; its device allocations are
// appended to `owned` (freed by whoever owns that list).
// With idx (the CSR's neighbour lists) and a_max <= 4 (b_max <= 16) the
// plan also packs the class-A (class-B) rows' neighbours next to their items
// (a_members, b_members), so that a gather reads a short row's descriptor
// and neighbours in one step.
int build_split_plan(hnv_graph* g, std::vector<void*>* owned, const int32_t* ptr, int32_t rows,
                     SplitPlan* plan, cudaStream_t s, const PlanShape& shape = PlanShape(),
                     const int32_t* idx = nullptr);
// Panel plan: the rows of `base` no longer than its class C bound keep their
// classes and items; the longer rows (listed ascending neighbour IDs in
// [0, cols)) are cut where their neighbours cross a panel boundary (P equal
// ranges of IDs) and into chunks of at most T incidences, and their items
// are listed panel by panel after the short classes, so that the launch
// over them works through the neighbour table one panel at a time (a
// panel's rows are read from DRAM about once and then hit L2). A long row
// left in one piece is a row item (n_d counts them); the pieces of a cut
// row are reduced in order (panel, then position) by the split-row
// reduction. P is chosen from table_bytes (the neighbour table's size) and
// the long rows' lengths; *panels = 1 means no panel plan (plan untouched).
int build_panel_plan(hnv_graph* g, std::vector<void*>* owned, const SplitPlan& base,
                     const int32_t* ptr, const int32_t* idx, int32_t cols, int64_t table_bytes,
                     SplitPlan* plan, int* panels, cudaStream_t s);
// The plan of one side of a level (0 hyperedge rows, 1 node rows) for
// neighbour rows of row_bytes: its panel plan (built on first use) or the
// regular one. HNV_PANELS=<k> forces k panels wherever there are long rows.
int side_plan(hnv_graph* g, Level* lv, int side, size_t row_bytes, const SplitPlan** plan,
              cudaStream_t s);
void free_level(Level* lv, cudaStream_t s);
int level_alloc(Level* lv, void** p, size_t bytes, cudaStream_t s);

// coarsen.cu: one step of Algorithm 1.
int coarsen_step(hnv_graph* g, int level, const hnv_coarsen_params* p, const uint64_t* d_explicit,
                 Level* fine, Level* coarse);

// refine.cu
// Scratch of `need` bytes for a call on s: *keep (*have bytes, the graph's),
// grown if it must be. In a capture, where memory allocated now is valid in the
// replays only, a larger one comes from the call's pool instead.
int graph_scratch(hnv_graph* g, float** keep, size_t* have, size_t need, TempPool& pool,
                  float** out, cudaStream_t s);
// dtype: HNV_F32 or HNV_BF16 row storage (sums in float32 either way).
int refine_level(hnv_graph* g, int level, void* z_v, void* z_e, int dtype, int d, float omega,
                 int sweeps, int mode, cudaStream_t s);
// One sweep from (v_in, e_in) into the buffers (v_out, e_out) (no overlap).
int refine_sweep_into(hnv_graph* g, int level, const void* v_in, const void* e_in, void* v_out,
                      void* e_out, int dtype, int d, float omega, int mode, cudaStream_t s);
int project_level(const hnv_graph* g, int fine_level, const void* zc_v, const void* zc_e,
                  void* zf_v, void* zf_e, int dtype, int d, cudaStream_t s);
// Sweeps until the largest change of any coordinate in a sweep is <= eps, or
// max_sweeps (synchronises after every sweep to read that change).
int refine_level_until(hnv_graph* g, int level, void* z_v, void* z_e, int dtype, int d,
                       float omega, int max_sweeps, float eps, int mode, int32_t* sweeps_done,
                       float* last_delta, cudaStream_t s);
// adjoint.cu: weights from a level-0 weight vector (device) to every level,
// and the reverse mode of the two-phase float32 V-cycle.
int set_weights_impl(hnv_graph* g, const float* d_w0, cudaStream_t s);
int vcycle_backward_impl(hnv_graph* g, const float* ckpt, const float* g_v0, const float* g_e0,
                         float* grad_w0, float* grad_zc, int d, float omega, int sweeps,
                         cudaStream_t s);

// tma_refine.cu: TMA-gather half-sweep for d in {32, 64, 128, 256}.
bool tma_supported(int d);
// One bounded mbarrier wait that nothing completes; sets ERRBIT_TIMEOUT in
// *err once it gives up after limit_ns.
int wait_selftest(int32_t* err, uint64_t limit_ns, cudaStream_t s);
int tma_half_sweep(const SplitPlan& plan, const int32_t* idx, const float* inc_w,
                   const float* inv_norm, const float* src, int64_t src_rows, const float* self_in,
                   float* out, int64_t self_rows, int d, float omega, float* partials,
                   int32_t* err, cudaStream_t s);

// General float32 row gather over a plan (used by the adjoint):
// out[r] = keep * self[r] + scale * norm[r] * sum_k wgt[k] * src[idx[k]];
// norm / wgt may be null (1); with keep == 0 self is not read. With conc, a
// graph with side streams, the plan's row classes run concurrently on them.
int gather_rows_f32(const SplitPlan& plan, const int32_t* idx, const float* wgt,
                    const float* norm, const float* src, const float* self_in, float* out, int d,
                    float keep, float scale, float* partials, cudaStream_t s,
                    const hnv_graph* conc = nullptr);

// team.cu: whole V-cycles or sweeps of small graphs in one cooperative launch.
// One side of a level for the team kernel: its regular plan (rows of 1-16
// incidences first) and arrays.
struct TeamSide {
  const int4* items = nullptr;
  const int4* long_desc = nullptr;
  const int32_t* idx = nullptr;
  const float* inc_w = nullptr;
  const float* inv_norm = nullptr;
  // items [0, n_a): rows of 1-4 incidences; [n_a, n_short): of 5-16; [n_short, n_rows): longer
  // whole rows; [n_rows, n_items): chunks, the n_mid rows' n_mid_chunks first
  int32_t n_a = 0, n_short = 0, n_rows = 0, n_items = 0, n_mid = 0, n_huge = 0, n_mid_chunks = 0;
};

struct TeamLevel {
  TeamSide side[2];               // 0 hyperedge rows, 1 node rows
  const int32_t* rep_v = nullptr;
  const int32_t* rep_e = nullptr;
  int32_t n = 0, m = 0;
  int64_t row0 = 0;               // rows of the finer levels (checkpoint offset)
};

// Levels top .. bottom of one graph: the rows start from zc (null: they are
// in place), level `bottom` is refined in zv0 / ze0, a level l above it in
// buf[l & 1] (node rows, then hyperedge rows).
struct TeamGraph {
  const TeamLevel* levels = nullptr;   // device
  int32_t top = 0, bottom = 0;
  const uint4* zc = nullptr;
  uint4* zv0 = nullptr;
  uint4* ze0 = nullptr;
  uint4* buf[2] = {nullptr, nullptr};
  float* partials = nullptr;
  uint4* jtmp = nullptr;               // Jacobi: m rows of the largest level
  uint4* ckpt = nullptr;               // every level's starting rows, or null
  int32_t* err = nullptr;              // the graph's error word
  uint64_t wait_ns = kTeamWaitNs;      // limit of a barrier wait
  int32_t stop_at = 0;                 // self-test: the barrier that is never complete, or 0
};

struct TeamArgs {
  TeamGraph one;                       // with graphs == null: one graph, one team
  const TeamGraph* graphs = nullptr;   // device: graphs of team t are
  const int32_t* team_first = nullptr; //   [team_first[t], team_first[t + 1])
  int32_t blocks = 1;                  // blocks per team
  int32_t dv = 0, sweeps = 0, jacobi = 0;
  float keep = 0.f, omega = 0.f;
  uint32_t* barriers = nullptr;        // 32 words per team, zeroed before the launch
  // stopping rule (result != null): delta holds 3 words, zeroed before the
  // launch; result (zeroed too) receives {sweeps done, bits of the last largest
  // change, ERRBIT_TIMEOUT if a wait gave up}
  unsigned* delta = nullptr;
  int32_t* result = nullptr;
  float eps = 0.f;
};

// Levels the team kernel can take: rows of at most 64 vectors, and so little
// work per half-sweep that launches, not bandwidth, may set its time. The
// stopping rule takes it for all of these: a launch per half-sweep also reads
// both tables again and the host waits every sweep (1.05-3 times slower on
// every level measured, 35 levels of 4 to 1,000K rows, 8 to 1,024 bytes a row).
constexpr int64_t kTeamMaxRowBytes = 1024;
constexpr int64_t kTeamMaxGather = 192000000;   // bytes gathered per half-sweep
constexpr int64_t kTeamMaxRows = 96000000;      // bytes of both row tables
constexpr int kTeamMaxSweeps = 512;             // of one launch
bool team_fits(const Level& lv, int dtype, int d);
// Levels of a fixed number of sweeps that it also runs faster than a launch per
// row class does (team.cu).
bool team_pays(const Level& lv, int dtype, int d);
void team_level(const Level& lv, int64_t row0, TeamLevel* out);
// Blocks that the items of one level's larger side fill.
int team_blocks_for(const Level& lv, int dtype, int d);
// Estimated microseconds of one sweep of a level by a team of `blocks` (to deal
// a batch's graphs over teams).
double team_sweep_us(const Level& lv, int dtype, int d, int blocks);
// Estimates to choose a batch's path by, fitted to the same batches (team.cu): a
// sweep of a level by a team of `blocks` of the device's SMs; a sweep each of
// `steps` steps of the step lists with `nnz` incidences in all.
double team_batch_us(const Level& lv, int dtype, int d, int blocks);
double step_batch_us(int steps, int64_t nnz, int dtype, int d);
// kTeamRefused: the device would not run the blocks at once (it has fewer SMs
// for this process than it says, or no cooperative launches), and nothing was
// launched; the caller takes the per-launch path.
constexpr int kTeamRefused = 1;
bool team_refused(cudaError_t e);   // the error that says so
int team_launch(TeamArgs a, int teams, int dtype, int d, cudaStream_t s);
// The team path applies at all (it is off while phases are timed, and where
// an environment switch asks for another gather).
bool team_enabled(int d);
// Levels top .. bottom of g (all of which fit) in one launch on s, or
// kTeamRefused.
// With eps, the stopping rule: the sweeps done, the last change and whether a
// wait gave up are left at *result (device; until the next launch on s).
int team_run(hnv_graph* g, TeamGraph t, int dtype, int d, float omega, int sweeps, int mode,
             cudaStream_t s, const float* eps = nullptr, const int32_t** result = nullptr);
// Uploads the TeamLevels of g's levels (from *host, which has to last until the
// graph's stream is next synchronised; the calls that build levels end with
// that, so later calls on any stream find them). Without memory for them
// g->team_levels stays null, and the per-launch path is taken.
void team_upload(hnv_graph* g, std::vector<TeamLevel>* host);
void team_drop(hnv_graph* g);   // the descriptors of a hierarchy that goes
inline bool team_ready(const hnv_graph* g) { return g->team_levels != nullptr; }
int forced_panels();   // HNV_PANELS, or -1

// Two-phase sweeps whose split-row partial sums go to caller-provided
// scratch (at least max(planE.n_chunks, planV.n_chunks) * d floats); no
// allocation and no timing events.
int refine_two_phase_with_partials(const hnv_graph* g, int level, float* z_v, float* z_e, int d,
                                   float omega, int sweeps, float* partials, cudaStream_t s);

// Reads the device error word (synchronising s) and clears it.
int read_and_clear_err(hnv_graph* g, cudaStream_t s, int32_t* bits);
// Copies `count` device ints into the graph's pinned buffer and synchronises.
int read_ints(hnv_graph* g, const int32_t* d_src, int count, int32_t* host_out, cudaStream_t s);

}  // namespace hnv
