// Internal state and helpers of libcb (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>

#include "cb.h"

namespace cb {

// Device-side error codes latched in Graph::err (first one wins).
enum DevErr : int32_t {
  kErrNone = 0,
  kErrRowLength = 1,     // a rebuilt row does not match the degree
  kErrValidate = 3,      // input graph not simple / symmetric / in range
  kErrResolve = 5,       // a dependency wait of the in-order pass gave up
  kErrStage = 6,         // a bulk copy into shared memory did not complete in time
  kErrUniform = 7,       // uniform trades: an inbox or the run queue overflowed, or a message missed its trade
  kErrUniformWait = 8,   // uniform trades: a wait for a queued trade or an inbox entry gave up
};
// The codes that report a bounded wait running out (CB_ETIMEOUT).
inline bool is_timeout(int32_t e) { return e == kErrResolve || e == kErrStage || e == kErrUniformWait; }

struct UniBufs;        // uniform-trade buffers (uniform.cu)
struct PresenceBufs;   // edge presence record (autocorr.cu)

constexpr int kBucketCapMax = 4096;  // largest "bucket_cap"
constexpr int kTileMaxCap = 128;    // largest trade (deg u + deg v) on the flat tile path
constexpr int kBlockMaxCap = 2048;  // largest trade on the 256-thread path
constexpr int kBlockMaxDefault = 1024;   // default of the "block_max" option
constexpr int kSmemMaxCap = 8192;   // largest trade kept in shared memory on the 1024-thread path
constexpr int kCounters = 64;       // device counters of one super step (two sets per handle, used in turn)
// Trade size classes of the threshold phase (one team size each) and the
// device counters of a super step.
constexpr int kClasses = 9;
constexpr int kClassLists = (kClasses + 1) / 2;   // arrays of their lists, two classes to each
constexpr int kWarpClasses = 3;     // classes 0..2 run on warps or parts of a warp
constexpr int kCtrClsLen = 0;       // [0, kClasses): trades per class
constexpr int kCtrFirstEnt = 10;    // [10, 10 + kClasses): their directed entries
constexpr int kRetryPassesMax = 4;
constexpr int kCtrDef = 24;         // [24 + 3 r, 27 + 3 r): trades that pass r deferred, by kind (r <= kRetryPassesMax)
constexpr int kCtrFinished = 40;    // chunks of the in-order pass claimed
constexpr int kCtrChunks = 41;      // its chunks
constexpr int kCtrClaim = 42;       // [42 + 3 r, 45 + 3 r): trades of each list that retry pass r claimed
static_assert(24 + 3 * (kRetryPassesMax + 1) <= 40 && 42 + 3 * kRetryPassesMax <= kCounters - 1, "counter layout");
constexpr int64_t kFuseMax = int64_t(1) << 17;    // trades from which the first pass has a kernel per class
constexpr int64_t kRetryMin = int64_t(1) << 20;   // trades from which retry passes run
constexpr int64_t kNarrowPackMax = int64_t(1) << 28;   // nodes up to which a far-trade record fits 8 bytes
constexpr int kRowChunk = 2048;      // entries per sample of the entry -> row index
constexpr int kScratch = 16;         // device words of a handle for creation and export
constexpr int kDefSegs = 1024;      // most segments of the trades that deferred ones are counted in
constexpr int kStats = 7 + 2 * kClasses;   // counters cb_stats reports
constexpr int kTimings = 6 + kClasses;     // values cb_timings reports
constexpr int kCtrGws = kCounters - 1;   // trades whose workspace is in global memory
constexpr int kMaxLcgGaps = 1024;   // p - n for the relaxed permutation (prime gaps below 2^31 are far smaller)

// One independent graph of a handle.  A plain handle holds one; a batch handle
// holds many side by side: graph i owns node ids and positions [off, off+span),
// and its keys use local ids and positions with its own seed and step, so it
// evolves exactly as it would alone.  An odd graph in a batch gets one padding
// node of degree 0 whose permutation key is the largest possible: it always
// takes the last position, and its trade with the node before it changes
// nothing, which is the untraded last position of an odd graph.
struct Seg {
  uint64_t seed;
  int64_t off;           // first node id (= first position)
  int64_t n;             // real nodes
  int64_t span;          // n, or n + 1 with a padding node
  int64_t bucket_base;   // first permutation bucket
  int64_t m;             // undirected edges
  int64_t pair_off;      // first exported pair
  int64_t slot_base;     // first id of its permutation bucket space
  uint32_t g;            // super step (advanced on the device at the end of each step)
  int32_t B;             // permutation bucket bits
  int32_t cap;           // ids one bucket holds
};

struct Graph {
  int64_t n = 0, nnz = 0, m = 0, T = 0, ntasks = 0;
  uint64_t seed = 0, g = 0;
  // segments (graphs) of the handle
  int nseg = 1;
  bool batch = false;             // made by cb_create_batch
  Seg* segs = nullptr;            // device table (nseg)
  int32_t* seg_of = nullptr;      // device: segment of each node id / position (null for a plain handle)
  Seg* hsegs = nullptr;           // host copy (g not kept current)
  int64_t nbuckets = 1;           // permutation buckets over all segments
  int32_t* pairs = nullptr;       // batch export: every graph's pairs, local ids
  uint64_t pairs_step = ~0ull;    // super step the pairs were exported at
  // CUDA graph of one super step per ping-pong parity
  bool use_graph = false;
  cudaGraphExec_t step_exec[2] = {nullptr, nullptr};
  int64_t step_launches = 0;      // kernels in one captured super step
  int64_t maxdeg = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int device = 0, num_sms = 0;

  // constant per graph
  int32_t* deg_id = nullptr;      // degree by node id
  int64_t* rp_id = nullptr;       // id-space row offsets (n+1)
  // per super step (ping-pong index `cur`)
  int cur = 0;
  int32_t* order[2] = {nullptr, nullptr};  // node at each position
  int64_t* rp[2] = {nullptr, nullptr};     // position-space row offsets (n+1)
  int32_t* chunk_row = nullptr;            // row of every kRowChunk-th entry of the offsets last computed
  int32_t* col[2] = {nullptr, nullptr};    // position-space rows, ascending
  int32_t* pos[2] = {nullptr, nullptr};    // position of each node (pos[1 - cur] is scratch between steps)
  int32_t* order2 = nullptr;               // third set (may_run_ahead(); else null): the step after next's, when
  int32_t* pos2 = nullptr;                 // computed ahead; then set 1 - cur is the next step's between steps
  int64_t* rp2 = nullptr;
  int32_t* chunk_row2 = nullptr;
  bool ahead = false;                      // set 1 - cur and the class lists are computed
  uint16_t* stash = nullptr;               // per placed entry (step g+1 layout): bit0 own flip, bits 1.. far key prefix
  uint64_t* thr_key = nullptr;             // per trade: threshold key
  uint64_t* thr_tb = nullptr;              // per trade: threshold tie-break (lo<<32|hi)
  uint32_t* done = nullptr;                // per trade: the step + 1 once its threshold is published
  uint64_t* far_pack = nullptr;            // per trade, 8 or (above kNarrowPackMax) 16 bytes: new positions of its nodes, threshold prefix (rebuild)
  void* far_wide = nullptr;                // 16-byte records in its place, where 8 would do ("wide_pack", tests)
  int32_t* lists = nullptr;                // kClassLists x ntasks: the trades of each size class (pair_lists.cuh)
  uint32_t* def_bits = nullptr;            // deferred trades, one bit each (zero between steps)
  int32_t* def_seg = nullptr;              // their counts per kind and segment (zero between steps)
  int32_t* def_list = nullptr;             // by kind for a retry pass; in index order with the chunks' first ones for the in-order pass
  int64_t* counters = nullptr;             // two sets of kCounters, then the CTAs that ended the step
  int32_t* err = nullptr;                  // latched device error
  int64_t* scratch = nullptr;              // kScratch words right after it
  void* arena = nullptr;                   // the allocation that holds the arrays above and below
  // workspaces
  void* ws_global = nullptr;               // global workspace for trades too big for smem
  size_t ws_slice = 0;                     // bytes per CTA slice
  int ws_ctas = 0;                         // number of slices
  char* sort_ws = nullptr;                 // permutation scratch
  char* scan_ws = nullptr;
  int64_t* host_counters = nullptr;        // host mirror of counters
  int64_t dev_bytes = 0, dev_bytes_peak = 0;   // device memory held by the handle

  // knobs
  int tile_max = kTileMaxCap;
  int tile_paths = 1;   // threshold phase of small trades: 1 one warp per trade, 0 256-thread CTAs
  int fix_passes = 0;   // passes of the rebuild's fix-up over slices of the far trades (0: sized for L2)
  int64_t fuse_max = kFuseMax, retry_min = kRetryMin;   // options, to test both sides on small graphs
  int fix_ctas = 0;             // test hook: CTAs of the rebuild (0: four per SM)
  int cta_paths = 1;    // threshold phase of larger trades: 1 register-resident CTA kernels, 0 shared-memory ones
  int cand_max = 32;    // register paths: candidates ranked directly (tests lower it to force radix digits)
  uint64_t wait_ns = 1000000000ull;       // longest single wait of a super step (dependency, bulk copy)
  uint64_t uni_wait_ns = 20000000000ull;  // longest single wait of the uniform-trade executor
  int hold_publish = 0;                   // test hook: trades never publish their done flags
  int inorder_ctas = 0;                   // test hook: CTAs of the in-order pass that take part (0: all)
  int64_t hold_trade = -1;                // test hook: uniform trade whose messages are dropped
  int block_max = kBlockMaxDefault;
  int smem_max = kSmemMaxCap;
  int bucket_cap = 2048;
  int inorder_threads = 1024;   // CTA size of the in-order threshold pass (256 or 1024)
  int retry_passes = 2;         // parallel passes over the deferred trades before the in-order pass
  int lane_teams = 1;           // trades up to 32 / 64 entries on teams of 8 / 16 lanes
  int uni_threads = 1024;       // CTA size of the uniform-trade executor (256, 512 or 1024)
  // relaxed global trade: permutations from h(x) = (a x + b) mod p
  bool relaxed = false;
  uint64_t lcg_p = 0;           // smallest prime >= n
  uint64_t* lcg_ab = nullptr;   // device: a, b of the step being prepared
  int64_t* lcg_gaps = nullptr;  // device: gap count, then the sorted gap values

  // uniform single trades (uniform.cu)
  UniBufs* uni = nullptr;
  uint64_t uni_next = 0;        // index of the next uniform trade
  // edge presence record for the autocorrelation of Section 5.1 (autocorr.cu)
  PresenceBufs* pres = nullptr;
  // swap counts (swaps.cu): device pair (performed, possible), when on
  bool swap_stats = false;
  int64_t* swaps = nullptr;

  // stats of the last cb_global_trades
  int64_t stats[kStats] = {0};
  int64_t launches = 0;                    // kernel launches issued by this handle
  bool timing = false;                     // record CUDA events around the phases
  // events, in two sets that super steps use in turn (the host waits for a
  // step's events only when the set comes round again, two steps later):
  // [0..4) phase bounds, [4, 4 + kClasses + 1) bounds of the first pass's
  // class kernels, then the end of the retry passes
  cudaEvent_t ev[2][4 + kClasses + 2] = {};
  int ev_set = 0;                          // the set the next super step records
  bool ev_pending[2] = {false, false};     // recorded, not yet added to phase_ms
  // permutation+prep, thresholds, rebuild, whole step, the first pass's
  // kernel of each size class, the retry passes, the in-order pass
  double phase_ms[kTimings] = {};
  int latched = CB_OK;
  std::string last_error;
};

inline int64_t next_pow2_host(int64_t x) {
  int64_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Records an error on the graph (or globally) and returns the code.
int fail(Graph* g, int code, const std::string& msg);
int cuda_fail(Graph* g, cudaError_t e, const char* what);

#define CB_CUDA(g, call)                                        \
  do {                                                          \
    cudaError_t e_ = (call);                                    \
    if (e_ != cudaSuccess) return ::cb::cuda_fail((g), e_, #call); \
  } while (0)

// Overlapped launches: step time without -> with, n=2^12 88 -> 80 us, 2^14 166
// -> 160, 2^15 187 -> 184, but 2^16 214 -> 219 and 2^18 436 -> 543 (waiting CTAs
// take the place of running ones).
constexpr int64_t kOverlapMax = int64_t(1) << 15;

// Overlapped launches (programmatic dependent launch): a kernel launched with
// overlap = true may be set up while the kernel before it in the stream still
// runs, so its launch costs no idle time; its first statement has to be
// after_previous(), which waits until that kernel has finished and its writes
// are visible.  Kernels that call before_next() let their successor be set up
// as soon as all their CTAs have started.  Without overlap both do nothing.
// A kernel with after_previous() is resident while the one before it still
// writes.  So it takes no __restrict__ pointers, and reads what earlier kernels
// write by plain loads or __ldcg, never __ldg: __restrict__ and __ldg both
// promise data that does not change while the kernel lives, and would let the
// compiler move a load above the wait.
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void before_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... P, class... A>
cudaError_t launch(bool overlap, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                   A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

// ---- kernels / host launchers implemented in the .cu files ----
// scan.cu
size_t scan_ws_bytes(int64_t n);
// out[0..n] = exclusive prefix sums of in[0..n), out[n] = total
cudaError_t exclusive_scan_i32(const int32_t* in, int64_t* out, int64_t n, void* ws, cudaStream_t s,
                               int64_t* launches = nullptr);

// Parts of a permutation: all of it, or, ahead of time, its scatter beside the
// end of the first pass (nothing where one kernel does it all) and the rest,
// with the class lists, beside the in-order pass.
enum class PermPart { kWhole, kScatterAhead, kRestAhead };

// permute.cu
struct ClassArgs;
size_t perm_ws_bytes(int64_t nbuckets, int64_t slots);
int bucket_bits(int64_t n);
int64_t bucket_space(int64_t span, int B);
// Does a handle of so many buckets, with so many keys to compute for all of
// them, take the one-kernel form?  (It needs no bucket space.)
bool perm_rescans(int64_t nbuckets, int64_t keys);
// order_out[p] = node at position p; pos_out[x] = position of x, rp_out[p] =
// row offsets of that order (n + 1; either may be null).  Each segment uses
// its device step counter + dg, or the step g_abs for all when g_abs >= 0.
// classes (may be null): build the size-class lists of the current step too.
int compute_permutation(Graph* h, uint32_t dg, int64_t g_abs, int32_t* order_out, int32_t* pos_out, int64_t* rp_out,
                        const ClassArgs* classes, PermPart part = PermPart::kWhole);
size_t perm_zero_bytes(int64_t nbuckets);   // the start of its scratch that has to be zero at first

// rows.cu
// dst row q <- src row rowmap[q] with values mapped through valmap (identity if null), ascending
int permute_rows(Graph* h, int64_t nrows, const int64_t* src_rp, const int32_t* src_col,
                 const int32_t* rowmap, const int32_t* valmap, const int64_t* dst_rp, int32_t* dst_col);
// Validation of the input: scan_rows checks ids and order and counts the
// entries on each side of the diagonal (synchronises); validate_sorted_graph
// then checks the symmetry of well formed rows and latches kErrValidate (not
// synchronising; `grouped` is scratch of row_ptr[n] int32).
struct Validation {
  char* ws = nullptr;          // graphs too large for L2: the partition's scratch
  size_t bytes = 0;
  int sh = 0, nb = 0, ctas = 0;
  int32_t* counts = nullptr;   // upper entries per (bucket, CTA)
  int64_t* place = nullptr;    // their exclusive scan
  void* scan = nullptr;
  int32_t err = 0;             // the device error word (kErrValidate: bad offsets)
  int64_t maxdeg = 0, upper = 0, lower = 0;
  bool unsorted = false;       // some row is not strictly increasing
  bool bad = false;            // an id out of range or a self loop
};
int scan_rows(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v);
int validate_sorted_graph(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v, int32_t* grouped);
void free_validation(Graph* h, Validation* v);
// like permute_rows without sorting (rows keep their order)
int relabel_rows(Graph* h, int64_t nrows, const int64_t* src_rp, const int32_t* src_col, const int32_t* rowmap,
                 const int32_t* valmap, const int64_t* dst_rp, int32_t* dst_col);
// canonical pairs (x < y, sorted, local ids) of the current step into `pairs`
// (2m int32, device); uses the spare adjacency buffer
int export_sorted_pairs(Graph* h, int32_t* pairs);

// trade.cu
// ahead: another step of the same call follows and compute its permutation
// beside this step's in-order pass (handles that runs_ahead() allows)
int super_step(Graph* h, bool ahead = false);
bool may_run_ahead(int64_t ntasks, int64_t nnz);
bool runs_ahead(const Graph* h);
int flush_timing(Graph* h, int set, bool add);   // wait for a recorded event set; add it to phase_ms
int init_trade_kernels(Graph* h);   // one-time kernel attributes (outside stream capture)
int init_perm_kernels(Graph* h);
size_t trade_ws_slice_bytes(int64_t max_trade);
bool runs_retries(const Graph* h);     // large enough for retry passes
int retry_passes_of(const Graph* h);   // retry passes a super step launches
bool small_handle(const Graph* h);     // launch-bound: its super steps use overlapped launches

// api.cu
// stream-ordered device allocation counted in the handle's device bytes
cudaError_t dev_alloc(Graph* h, void** p, size_t bytes);
// read the latched device error word (synchronises the stream)
int check_device_error(Graph* h);
// forget the recorded super-step graphs (they are recorded again when next needed)
void drop_step_graphs(Graph* h);

// swaps.cu
int count_swaps(Graph* h);                 // add the last super step's counts
int set_swap_stats(Graph* h, bool on);     // on: counts from zero

// uniform.cu
int uniform_trades(Graph* h, uint64_t count);
void free_uniform(Graph* h);

// autocorr.cu
int set_presence(Graph* h, int64_t T);   // T > 0: record the next T super steps (and now); 0: stop
int record_presence(Graph* h);           // the current state, while recording
void free_presence(Graph* h);

// device bytes a plain handle of n nodes / nnz entries / largest degree takes (upper estimate)
int64_t estimate_handle_bytes(int64_t n, int64_t nnz, int64_t maxdeg, int num_sms);
// record the CUDA graphs of the super step now (when the cuda_graph option is on)
int prepare_step_graphs(Graph* h);

}  // namespace cb

struct cb_graph : cb::Graph {};
