// context.h -- internal to the OASM library: the context a C-ABI handle
// points to, and the host-side helpers its translation units share
// (api.cu: the entry points; tables.cu: pattern tables; step.cu: planning,
// launching and finishing a batched step).  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <chrono>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <queue>
#include <string>
#include <vector>

#include "host_pool.h"
#include "kernels.h"

namespace oasm {

// NVTX range over a library call: named ranges for Nsight tools around feed,
// step and flush; without an attached tool a push/pop is a pointer test.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

constexpr size_t kFrontPad = 1024;   // arena bytes before the first work item
constexpr size_t kEndPad = 2048;     // arena bytes after the last one
constexpr size_t kChunk = 1 << 16;   // largest gather copy per block
constexpr size_t kShortChunk = 4096; // ... per warp, where no copy of a step is longer

struct Piece {
  bool dev;
  const uint8_t* dptr;  // device pointer (dev) or nullptr
  size_t host_off;      // offset into its pinned staging buffer (host pieces)
  size_t n;
  int sb = 0;           // staging buffer (host pieces)
};


// Vector storage that leaves new elements uninitialised: decided records are
// copied in right after the resize, so zero-filling them first would be a
// wasted pass over memory.
template <class T>
struct NoInitAlloc : std::allocator<T> {
  template <class U>
  struct rebind {
    using other = NoInitAlloc<U>;
  };
  NoInitAlloc() = default;
  template <class U>
  NoInitAlloc(const NoInitAlloc<U>&) noexcept {}
  template <class U>
  void construct(U* p) noexcept {
    ::new (static_cast<void*>(p)) U;
  }
  template <class U, class... Args>
  void construct(U* p, Args&&... args) {
    ::new (static_cast<void*>(p)) U(std::forward<Args>(args)...);
  }
};
using HitVec = std::vector<oasm_hit, NoInitAlloc<oasm_hit>>;

// Copies the pieces (dst, src, records) on up to 16 host threads, each
// thread taking an equal share of the bytes (pieces are cut where needed).
struct CopyTask {
  oasm_hit* dst;
  const oasm_hit* src;
  size_t n;
};
inline void parallel_copy(const std::vector<CopyTask>& tasks) {
  size_t total = 0;
  for (const CopyTask& t : tasks) total += t.n;
  const size_t T = std::max<size_t>(1, std::min<size_t>(16, total >> 18));
  parallel_parts(T, 1, [&](size_t t0, size_t t1) {
    for (size_t t = t0; t < t1; ++t) {
      const size_t lo = total * t / T, hi = total * (t + 1) / T;  // this share of records
      size_t pos = 0;
      for (const CopyTask& c : tasks) {
        const size_t a = std::max(lo, pos), b = std::min(hi, pos + c.n);
        if (a < b) memcpy(c.dst + (a - pos), c.src + (a - pos), (b - a) * sizeof(oasm_hit));
        pos += c.n;
        if (pos >= hi) break;
      }
    }
  });
}

struct StreamRec {
  bool open = false;
  bool clean = true;      // device windows of the slot are all empty
  int64_t pos = 0;        // symbols processed
  int32_t tail_len = 0;   // symbols of the stored tail
  bool eos_pending = false;
  std::vector<Piece> pieces;
  size_t pending = 0;
  HitVec ready;                 // decided hits; [head, end) not yet returned
  size_t head = 0;
  std::vector<size_t> runs;     // starts of canonically sorted runs in `ready`
  // A step's records of this stream, left where that step put them (one of
  // the context's two pinned record buffers, lent_buf) when the queue above
  // was empty: a drain or flush copies them out once instead of twice.  They
  // move into `ready` before that buffer is written again or before a later
  // step's records join them; while lent_n > 0, `ready` is empty.
  const oasm_hit* lent = nullptr;
  size_t lent_n = 0;
  int lent_buf = 0;
  // A fresh record that keeps the storage of its queue and its pieces (no new
  // pages to touch, no allocation per stream).
  void reset() {
    StreamRec fresh;
    ready.clear();
    pieces.clear();
    fresh.ready.swap(ready);
    fresh.pieces.swap(pieces);
    *this = std::move(fresh);
  }
};

// A finished step whose records are still on their way to the host: the
// copy into pinned buffer `buf` runs on the context's copy stream while the
// caller goes on (a next step may already run on the device).  The first
// call that needs the queues waits for it and hands the records to their
// streams (settle_records).
struct PendingRecords {
  bool on = false;
  bool direct = false;  // already in the pinned buffer (a small step wrote them)
  int buf = 0;
  size_t n = 0;
  std::vector<uint32_t> sids;                 // stream of each work item
  std::vector<unsigned long long> run_start;  // [items + 1] first record of each
};

inline bool canon_less(const oasm_hit& a, const oasm_hit& b) {
  if (a.pattern_id != b.pattern_id) return a.pattern_id < b.pattern_id;
  if (a.decided_at != b.decided_at) return a.decided_at < b.decided_at;
  if (a.k != b.k) return a.k < b.k;
  return a.len < b.len;
}

struct Bucket {
  int W = 0;
  int algo = 0;           // 0: Myers/Hyyro bit-vectors; 1 + K: automaton for K <= 3;
                          // kAlgoCut: multi-word Myers/Hyyro with the cut-off
  int max_nseg = 1;
  int warps = 8;          // warps per scan block
  int chunk = 1024;       // text bytes per TMA buffer (dictionary mapping)
  int gpw = 1;            // lane groups per warp (dictionary mapping, W = 1)
  double region_scale = 1.0;
  int kmax = 0;
  int ov_max = 1;
  std::vector<LaneGroup> groups;
  LaneGroup* d_groups = nullptr;
  uint32_t* d_peq = nullptr;
  uint32_t* d_peq_hi = nullptr;  // cut-off classes: the whole W-word table (d_peq: word 0)
  // weighted path (algo == kAlgoWeighted): per group (one warp's column of
  // 32 x kWRows rows holding several patterns) one 32-bit row word per row,
  // lane-major (lane l holds rows kWRows l .. kWRows l + kWRows - 1); see
  // kWildRow / kWFirstLane for the fields
  uint32_t* d_wrow = nullptr;
};

template <class T>
struct DevArray {
  T* p = nullptr;
  size_t cap = 0;  // elements
};

// The gram index (grams.cu) of a context: its tables, and the buckets of the
// patterns that stay on the forward scan while it runs.  It also takes the
// piece filter's patterns; if it cannot take all of them the piece filter runs
// beside it (both put their ends through one set).
struct Grams {
  uint32_t n_pat = 0;         // patterns it serves; 0: no index
  GramTables t{};
  GramScan scan{};            // tables; a step adds its text and buffers
  double rate = 0;            // expected suspects per text symbol
  double looks = 0;           // expected entries compared per text symbol,
  double most_looks = 0;      // and the most that any text can cause
  double clk = 0;             // clocks of an SM per symbol it takes
  double saved_clk = 0;       // and saves, against the forward scan of every pattern
  bool all_pref = false;      // serves every pattern of the piece filter
  std::vector<Bucket> rest;
  DevArray<unsigned long long> susp;
  DevArray<unsigned long long> longs;
  DevArray<GramCounters> ctr;
  int off_steps = 0;          // steps left without the index (suspects too dense)
};

// Where a step's launches begin: at its text, or, after a small step that left
// its launch, at the verification or at the sort.
enum { kFromText = 0, kFromCandidates, kFromHits };

// Bounds that tests lower to reach what lies behind them (oasm_selftest_limits).
struct Limits {
  // A small step of more candidates or hits goes on as separate launches.  In a
  // text of one repeated symbol all hits of a pattern are one chain that a
  // thread walks at 175 ns a hit (46 ms for so many), while the others wait at a
  // barrier, for a second or more: 33 M hits in 1 MiB ran out of that wait.  The
  // separate launches are as fast by then (a motif of 8 symbols, K = 3: 212,000
  // hits 171 us a step here and 208 there, 424,000 238 and 233, 844,000 369 and
  // 288).
  unsigned long long small_cand = 1ull << 22, small_hits = 1ull << 18;
  BarrierBound barrier;
  size_t gram_slice = size_t(1) << 27;  // arena symbols per slice of suspects
};

struct StepPlan {
  std::vector<WorkItem> items;
  std::vector<uint32_t> sids;
  std::vector<size_t> take;
  std::vector<Region> regions;       // all buckets, concatenated
  std::vector<size_t> region_off;    // per bucket
  std::vector<CopyChunk> chunks;
  size_t arena_bytes = 0;
  size_t longest_chunk = 0;
  int sb = 1, kb = 10;
  uint64_t new_bytes = 0;
  bool ordered = false;              // records written in canonical order (no record sort)
  bool small = false;                // everything after the candidates in one launch
  bool no_small = false;             // ... not again: that launch left the step
  int from = kFromText;              // where the launches of the step begin
  size_t set_len = 0;                // slots of the (end, pattern) set it uses
  bool grams = false;                // the gram index and the rest buckets scan this step
  // An empty plan that keeps its vectors' storage.
  void clear() {
    StepPlan fresh;
    const auto keep = [](auto& to, auto& from) {
      from.clear();
      to.swap(from);
    };
    keep(fresh.items, items);
    keep(fresh.sids, sids);
    keep(fresh.take, take);
    keep(fresh.regions, regions);
    keep(fresh.region_off, region_off);
    keep(fresh.chunks, chunks);
    *this = std::move(fresh);
  }
};

// Pinned host staging for fed bytes, with its device copy.  Two of them
// alternate: bytes fed while a step is in flight go to the buffer that step
// does not read, and a buffer is reused from its start once every piece in
// it has been consumed.
struct Stage {
  uint8_t* h = nullptr;
  size_t cap = 0, used = 0;
  size_t pending = 0;    // bytes of pieces still waiting for a step
  size_t copied = 0;     // bytes [0, copied) already on the device
  DevArray<uint8_t> d;
};

// A step launched by oasm_step_begin and not yet finished.
struct Flight {
  bool on = false;
  StepPlan pl;
  const WorkItem* d_items = nullptr;
  const Region* d_regions = nullptr;
  const CopyChunk* d_chunks = nullptr;
};

}  // namespace oasm

using namespace oasm;

struct oasm_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  oasm_config cfg{};
  Rules rules{};
  std::string err;
  int num_sms = 152;

  uint32_t n_pat = 0;
  std::vector<std::vector<uint8_t>> pats;
  std::vector<uint8_t> m, K;
  std::vector<uint32_t> mem_off;
  uint32_t mem_stride = 0;
  int T = 1;
  int kmax = 0;
  uint8_t* d_m = nullptr;
  uint8_t* d_K = nullptr;
  uint32_t* d_mem_off = nullptr;
  uint32_t* d_peq_rev = nullptr;
  // integer edit costs (oasm_create_weighted): the weighted dynamic program
  // replaces the bit-parallel scan and verification
  bool weighted = false;
  oasm_costs costs{1, 1, 1};
  uint8_t* d_bytes = nullptr;  // [n_pat][OASM_MAX_PATTERN_LEN] pattern symbols
  std::vector<Bucket> buckets;
  // piece filter (cfg.prefilter_piece): tables of the patterns it serves
  std::vector<char> on_filter;  // per pattern
  uint32_t n_pref_pat = 0;
  PrefSlot* d_pdir = nullptr;
  uint32_t pdir_bits = 0, pmax_probe = 0;
  uint32_t* d_pbloom = nullptr;
  uint32_t pbloom_bits = 0;
  PrefEntry* d_pent = nullptr;
  uint8_t* d_pbytes = nullptr;
  uint32_t* d_poff = nullptr;
  DevArray<unsigned long long> pset;  // (end, pattern) set, capacity a power of two
  double set_rate = 1.0 / 16;         // slots per symbol of a step's text
  Grams grams;

  // streams
  std::vector<StreamRec> streams;
  // host ranges registered for zero-copy feeds (read by the gather kernel
  // over the CPU-GPU link instead of through pinned staging)
  struct HostRange {
    const uint8_t* host;
    size_t bytes;
    const uint8_t* dev;
  };
  std::vector<HostRange> host_ranges;
  // free slots, lowest first (a stream takes the lowest free slot)
  std::priority_queue<uint32_t, std::vector<uint32_t>, std::greater<uint32_t>> free_slots;
  uint8_t* d_tails = nullptr;
  WinHdr* d_hdr = nullptr;
  MemRow* d_mem = nullptr;
  size_t stream_bytes = 0;
  uint32_t n_open = 0;
  Flight flight;
  bool debug = false;

  // host staging (pinned)
  Stage stage[2];
  int cur_stage = 0;         // the buffer new host bytes go to
  size_t stage_limit = size_t(2) << 30;

  // step buffers
  DevArray<uint8_t> arena, upload;
  DevArray<Candidate> cand;
  DevArray<unsigned long long> keys, keys_alt;
  DevArray<DevHit> out;
  // canonically ordered records, two buffers: a step writes rec_buf while the
  // previous step's records may still be copied out of the other
  DevArray<DevHit> out_sorted[2];
  int rec_buf = 0;
  PendingRecords pend;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t copy_done[2] = {};
  DevArray<unsigned long long> okeys, okeys_alt;
  DevArray<uint32_t> ovals, ovals_alt;
  DevArray<WinHdr> pool_hdr;
  DevArray<MemRow> pool_mem;
  DevArray<uint32_t> pool_pair;
  DevArray<int32_t> pair_pool;
  DevArray<DevHit> rtmp;             // ordered records by segment position
  DevArray<uint32_t> seg;             // segment counts, then output offsets
  DevArray<unsigned long long> seg_part;  // the scan's per-block sums
  DevArray<unsigned long long> run_start;  // [n_items + 1] records of each work item
  unsigned long long* h_run_start = nullptr;  // pinned copy, read after the step
  size_t h_run_start_cap = 0;
  StepCounters* d_ctr = nullptr;
  StepCounters* h_ctr = nullptr;
  unsigned int* d_hist = nullptr;
  uint8_t* h_upload = nullptr;
  size_t h_upload_cap = 0;
  DevHit* h_out[2] = {};      // pinned record buffers, one per out_sorted buffer
  size_t h_out_cap[2] = {};
  cudaEvent_t ev[9] = {};  // 0-5 step phases, 6-7 autotune, 8 piece filter start
  cudaEvent_t done = nullptr;
  cudaEvent_t staged = nullptr;  // host staging copies of the step in flight done
  // executable step graphs, one per step topology (which kernels a step
  // launches: its scan classes, the piece filter, the gram index, the record
  // order), each updated in place while its topology repeats; the least
  // recently used one is dropped when a new topology needs a slot
  struct GraphSlot {
    uint64_t topo = 0;
    uint64_t used = 0;
    cudaGraphExec_t exec = nullptr;
  };
  static constexpr size_t kGraphSlots = 8;
  std::vector<GraphSlot> graphs;
  uint64_t graph_clock = 0;
  uint64_t step_topo = 0;    // topology of the step being enqueued
  int small_blocks = 0;      // blocks of the small steps' launch (0: it does not fit
                             // the device, and no step is launched so)
  int sort_blocks = 0;       // radix-sort blocks: as many as are resident together
  bool capturing = false;

  oasm_stats st{};
  oasm_routes routes{};
  Limits limits;
  bool many_hits = false;    // the last step of a small step's size went over them
  uint64_t fingerprint = 0;  // patterns, thresholds and rules (stream checkpoints)
};

namespace oasm {

int fail(oasm_ctx* c, int code, const char* fmt, ...);
int ensure_host(oasm_ctx* ctx, uint8_t** p, size_t* cap, size_t n, size_t keep);
// Output record buffers for n records; `ordered` steps need only the
// canonically ordered one.
int ensure_out(oasm_ctx* ctx, size_t n, bool ordered = false);
int ensure_pool(oasm_ctx* ctx, size_t n);  // room for n windows that a step leaves
int bits_for(uint64_t v);  // bits needed to hold 0..v

int wait_event(oasm_ctx* ctx, cudaEvent_t ev);
void free_ctx(oasm_ctx* c);
int build_prefilter(oasm_ctx* ctx, const std::vector<char>& pref);
int build_tables(oasm_ctx* ctx);
// The gram index: with no device memory for all of it there is none, and it gives
// its own to what the context cannot do without (must_alloc).  It is built before
// the stream state, not after: its directory lies better there (a scan of 32 MiB
// of bytes 125 us, and 128 where it came last).
int build_index(oasm_ctx* ctx);
void drop_grams(oasm_ctx* ctx);  // frees the index and its buffers
void free_buckets(std::vector<Bucket>& bs);
// cudaMalloc (that oasm_selftest_alloc can let fail).
cudaError_t dev_alloc(void** p, size_t bytes);
template <class T>
cudaError_t dev_alloc(T** p, size_t bytes) {
  return dev_alloc(reinterpret_cast<void**>(p), bytes);
}
// dev_alloc; without memory for it the gram index gives up its own.
template <class T>
cudaError_t must_alloc(oasm_ctx* ctx, T** p, size_t bytes) {
  cudaError_t e = dev_alloc(p, bytes);
  if (e == cudaErrorMemoryAllocation && ctx->grams.n_pat) {
    cudaGetLastError();
    drop_grams(ctx);
    e = dev_alloc(p, bytes);
  }
  return e;
}
// Tables of the gram index; served[p] = 1 for the patterns it takes (all 0
// when it would not pay).
int build_grams(oasm_ctx* ctx, const std::vector<char>& pref, std::vector<char>& served);
void finish_grams(oasm_ctx* ctx);
double group_cost(int W, int algo);
void choose_piece_filter(const uint8_t* const* pat, const uint32_t* len, const uint32_t* k,
                         uint32_t n, uint32_t piece, uint8_t* on_filter);
StepParams make_params(oasm_ctx* ctx, const WorkItem* d_items, uint32_t n_items, int sb, int kb,
                       bool ordered = false);
// Chooses whether the step writes its records in canonical order and sizes
// the buffers that path needs.
int prepare_records(oasm_ctx* ctx, StepPlan& pl);
int bucket_gpw(const oasm_ctx* ctx, const Bucket& b);
int64_t region_len(oasm_ctx* ctx, const Bucket& b, int64_t total_ends);
int plan_step(oasm_ctx* ctx, StepPlan& pl);
void plan_regions(oasm_ctx* ctx, StepPlan& pl);
// The buckets a step scans: all, or those of the patterns the gram index leaves.
inline std::vector<Bucket>& step_buckets(oasm_ctx* ctx, const StepPlan& pl) {
  return pl.grams ? ctx->grams.rest : ctx->buckets;
}
cudaError_t record_event(oasm_ctx* ctx, cudaEvent_t e, cudaStream_t s);
int enqueue_step(oasm_ctx* ctx, StepPlan& pl, const WorkItem* d_items, const Region* d_regions,
                 const CopyChunk* d_chunks);
double ms_since(std::chrono::steady_clock::time_point t0);
int launch_step(oasm_ctx* ctx);
int finish_step(oasm_ctx* ctx, StepPlan& pl, const WorkItem* d_items, bool* overflow);
// Waits for the records of the last finished step to reach the host and
// hands them to their streams' queues (no-op when none are on the way).
int settle_records(oasm_ctx* ctx);
void release_stages(oasm_ctx* ctx);
int step_begin(oasm_ctx* ctx);
int step_end(oasm_ctx* ctx);
int run_step(oasm_ctx* ctx);
uint64_t fnv1a(uint64_t h, const void* p, size_t n);
size_t state_bytes(const oasm_ctx* ctx);
int check_sid(oasm_ctx* ctx, uint32_t sid);

#define CK(call)                                                                        \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ == cudaErrorMemoryAllocation) cudaGetLastError();                            \
    if (e_ != cudaSuccess)                                                              \
      return fail(ctx, e_ == cudaErrorMemoryAllocation ? OASM_ENOMEM : OASM_ECUDA,      \
                  "%s failed: %s", #call, cudaGetErrorString(e_));                      \
  } while (0)

// Room for n elements (the old contents are not kept).  Without device memory
// for it the gram index gives up its own, unless the room is for the index: a
// step planned with it is planned again (launch_step).
template <class T>
int ensure(oasm_ctx* ctx, DevArray<T>& a, size_t n, const char* what, bool for_index = false) {
  if (a.cap >= n && a.p) return OASM_OK;
  size_t want = std::max<size_t>(n, a.cap + a.cap / 2);
  want = std::max<size_t>(want, 1024);
  if (a.p) cudaFree(a.p);
  a.p = nullptr;
  a.cap = 0;
  ctx->st.buffer_grows += 1;
  const cudaError_t e = for_index ? dev_alloc(&a.p, want * sizeof(T))
                                  : must_alloc(ctx, &a.p, want * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    a.p = nullptr;
    return fail(ctx, OASM_ENOMEM, "device allocation of %zu bytes for %s failed: %s",
                want * sizeof(T), what, cudaGetErrorString(e));
  }
  a.cap = want;
  return OASM_OK;
}

// A power-of-two capacity of at least n (the piece filter's open-addressing set).
template <class T>
int ensure_pow2(oasm_ctx* ctx, DevArray<T>& a, size_t n, const char* what,
                bool for_index = false) {
  if (a.p && a.cap >= n) return OASM_OK;
  size_t want = 1024;
  while (want < n || want < 2 * a.cap) want <<= 1;
  return ensure(ctx, a, want, what, for_index);
}

}  // namespace oasm
