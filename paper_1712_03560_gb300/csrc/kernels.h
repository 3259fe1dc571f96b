// kernels.h -- host-side launchers of the OASM device path.  Internal.
#pragma once
#include <cuda_runtime.h>

#include "oasm_internal.cuh"

namespace oasm {

// Forward scan (Sellers search, bit-parallel) over one word-count class.
struct ScanArgs {
  const LaneGroup* groups;   // [n_groups]
  const uint32_t* peq;       // [n_groups][256 symbols][W words][32 lanes]; automaton
                             // classes of K = 2: [n_groups][256][B, B >> 1][32]
  int32_t n_groups;
  int32_t W;
  const Region* regions;     // [n_regions]
  int32_t n_regions;
  int32_t warps;             // warps per block
  int32_t resv;              // candidate slots a warp reserves at a time
  int32_t dict;              // 1: dictionary mapping (one pattern per lane, nseg = 1)
  int32_t chunk;             // text bytes per TMA buffer (dictionary mapping)
  int32_t algo;              // 0: Myers/Hyyro bit-vectors; 1 + K: automaton for K <= 3 (W = 1);
                             // kAlgoCut: Myers/Hyyro with the cut-off (W >= 2)
  int32_t gpw;               // lane groups per warp: 1, or 2 (dictionary mapping, W = 1)
  int32_t c_sub, c_ins, c_del;  // edit costs (algo == kAlgoWeighted)
  const uint32_t* wrow;      // weighted path: [n_groups][32 kWRows] row words, lane-major
  const uint32_t* peq_hi;    // cut-off classes: [n_groups][256][W][32] in global memory
                             // (peq then holds word 0 only: [n_groups][256][32])
  const WorkItem* items;
  const uint8_t* arena;
  Candidate* cand;
  unsigned long long cap_cand;
  StepCounters* ctr;
  uint32_t two;              // 2, and the bytes of one symbol's Peq row, as kernel
  uint32_t row_bytes;        // arguments (set by the launchers; see fma_dbl in scan.cu)
  uint32_t half;             // 2^31 (see half_plus in scan.cu)
};

// Weighted dynamic program over patterns' rows (oasm_create_weighted).  A
// group is one warp's column of 32 lanes x kWRows rows; patterns sit in runs
// of whole lanes, each ending at the last row of its last lane (rows above a
// pattern in its first lane are wild).  A row word holds the pattern symbol
// (bits 0-7), kWildRow, the row's index within its pattern, 1-based
// (bits 16-23; 0 for a wild row), and kWFirstLane on every row of a
// pattern's first lane (the row above that lane is Sellers' zero row).
constexpr int kAlgoWeighted = 8;
// Multi-word Myers/Hyyro classes with the cut-off of the blocks-based scan:
// only word 0 (pattern rows 1..32) runs while no lane's first 32 rows come
// within K of a match; see scan.cu.  Rows are low-aligned (row r at bit r - 1).
constexpr int kAlgoCut = 9;
constexpr int kWRows = 4;
constexpr uint32_t kWildRow = 0x100u;
constexpr uint32_t kWFirstLane = 1u << 24;

// Words per symbol row of a class's staged table: W for the Myers/Hyyro
// classes, word 0 only for the cut-off classes, the match mask B for the
// automaton classes of K = 0 and 1, and B and B >> 1 for those of K = 2 and 3
// (see nfa_step in scan.cu).
inline int staged_words(int W, int algo) {
  return algo == kAlgoCut ? 1 : algo == 3 || algo == 4 ? 2 : (algo >= 1 && algo <= 2) ? 1 : W;
}

// Shared memory of one scan block: the Peq tables of its gpw lane groups (256
// rows of staged_words x 32 words each), two text buffers per warp
// (dictionary mapping) and the mbarriers.
inline size_t scan_smem_bytes(int W, int warps, int chunk, int gpw = 1, int algo = 0) {
  const int w = staged_words(W, algo);
  return size_t(256) * 128 * w * gpw + size_t(warps) * 2 * chunk + size_t(1 + 2 * warps) * 8;
}

cudaError_t launch_scan(const ScanArgs& a, cudaStream_t s);
// Raises the dynamic shared-memory limit of every scan kernel (once per
// context, outside any stream capture).
cudaError_t prepare_scan_kernels(int max_smem_bytes);

// Copies of stream bytes into the step's text arena.
struct CopyChunk {
  const uint8_t* src;
  uint64_t dst_off;
  uint32_t len;
  uint32_t pad;
};
// short_chunks: a warp per chunk instead of a block
cudaError_t launch_gather(const CopyChunk* chunks, int n, bool short_chunks, uint8_t* arena,
                          cudaStream_t s);

// Set of (arena offset of an end << 24 | pattern) keys; all ones = empty.
struct EndSet {
  unsigned long long* slots;
  unsigned long long mask;   // capacity - 1 (a power of two)
};

// Piece filter over segments of the step's text: exact matches of pattern
// pieces propose candidate ends, deduplicated through an open-addressing set.
struct PrefArgs {
  const PrefSlot* dir;
  uint32_t dir_bits;             // directory size 2^dir_bits
  uint32_t max_probe;            // longest probe sequence in the directory
  const PrefEntry* ent;
  const uint8_t* pbytes;         // all patterns' bytes
  const uint32_t* poff;          // [n_pat] first byte of each pattern in pbytes
  const Region* segs;            // text segments [a, b) of start positions
  int32_t n_segs;
  int32_t pad;
  EndSet set;
  const uint32_t* bloom;         // 2^bloom_bits bits: two hash bits per piece prefix
  uint32_t bloom_bits;
  int32_t grid;                  // resident blocks (each walks many segments)
  uint32_t dir_in_smem;          // 1: the directory (<= kPrefDirSmem bytes) is staged in
                                 // shared memory and the Bloom bits are skipped
  uint32_t pad2;
};
constexpr size_t kPrefDirSmem = 64 << 10;
constexpr int kPrefSegMax = 4096;  // start positions per segment
cudaError_t launch_prefilter(const StepParams& p, const PrefArgs& f, cudaStream_t s);
cudaError_t prepare_prefilter_kernel(int max_smem_bytes);

// Gram index in front of the forward scan (grams.cu).
constexpr int kGramThreads = 1024;            // threads of an index scan block (one per SM)
constexpr uint32_t kGramMaxWords = 45056;     // 176 KiB of table bits in shared memory
constexpr int kGramLens = 6;                  // key lengths of an index
// odd multipliers: table bits of hashed keys, directory
constexpr uint32_t kGramBitMul = 0x9E3779B1u, kGramDirMul = 0x2C1B3C6Du;
struct GramLen {             // one key length: the first symbols of a gram
  uint32_t mask;             // the key within 16 2-bit symbols, or four bytes
  uint32_t mul, shift;       // table bit of a key: (key * mul) >> shift
  uint32_t word0;            // first word of the length's table
  uint32_t dir0;             // first directory slot
  uint32_t dir_shift, dir_mask, max_probe;
};
constexpr int kGramPair = 8;  // symbols of a pair looked at beside a gram
constexpr int kGramLeft = 128, kGramEdit = 64;
struct GramEntry {           // one gram of a pattern
  uint32_t pat;              // pattern | K << 24 | most edits of an occurrence << 28
                             // (K under unit costs)
  uint8_t before, after;     // pattern symbols beside the part that the gram stands for
  uint8_t pair;              // symbols of its pair beyond the gram (at most kGramPair),
                             // kGramLeft: before it; kGramEdit: the gram holds an edit;
                             // bits 4-5: symbols of that part - len + 1
  uint8_t len;               // symbols of the gram
  uint32_t lo, hi;           // 16 2-bit symbols (lo), or eight bytes
};
struct GramCounters {        // one per slice of the arena
  unsigned long long n_susp;
  unsigned long long n_long[3];  // suspects left of patterns of two, three, four words
  unsigned long long n_look;     // entries compared with the text, where they are many
};
struct GramTables {
  const GramEntry* entries;
  const uint32_t* peq_fwd;   // [n_pat][256][4] forward match masks
  int32_t any_long;          // 1: a gram has more than 32 pattern symbols on a side
};
struct GramScan {
  GramLen len[kGramLens];
  int32_t n_len;
  int32_t two_bit;           // 1: symbols as (byte >> shift2) & 3
  uint32_t shift2;
  uint32_t n_words;          // table words (a multiple of 4)
  const uint32_t* bits;
  const uint4* dir;          // {key, first entry, entries (0 = empty), -}
  const GramEntry* entries;
  const uint8_t* arena;
  unsigned long long t_begin, t_end;  // 512-symbol tiles of this slice
  unsigned long long* susp;  // arena offset of a gram << 24 | entry
  unsigned long long cap_susp;
  unsigned long long* longs; // [3][cap_long] suspects left, by word count
  unsigned long long cap_long;
  GramCounters* ctr_slice;
  StepCounters* ctr;
  unsigned long long text_end;  // arena offset after the last item's text
  unsigned long long cap_look;  // entries compared before the text is too dense; 0: any
};
cudaError_t prepare_gram_kernels();
// Match masks [n_pat][256][4] from the patterns' bytes ([n_pat][128]): bit j
// of a row is symbol j, or the j-th from the end.
cudaError_t launch_peq(const uint8_t* bytes, const uint8_t* len, uint32_t n_pat, uint32_t* peq,
                       bool reversed, cudaStream_t s);
// scan, ends and long of one slice (two or three launches)
cudaError_t launch_grams(const StepParams& p, const GramTables& g, const GramScan& a,
                         const EndSet& set, cudaStream_t s);

cudaError_t launch_verify(const StepParams& p, cudaStream_t s);

// Bound of a wait at a grid barrier.  `extra` arrivals more than there are
// blocks are waited for: 0, or 1 in a self-test that lets the wait run out.
struct BarrierBound {
  uint32_t polls = 1u << 22;  // a second or more
  uint32_t extra = 0;
};

// Stable LSD radix sort (8-bit digits) of keys by bits [lo_bit, hi_bit),
// with an optional 32-bit payload, in one cooperative launch.  The element
// count is read on the device from *count (clamped to cap).  On return
// *keys_out / *vals_out point at whichever buffer of each pair holds the
// sorted data.
struct SortArgs {
  unsigned long long* keys;
  unsigned long long* keys_alt;
  uint32_t* vals;                 // may be null
  uint32_t* vals_alt;
  const unsigned long long* count;
  unsigned long long cap;
  int lo_bit, hi_bit;
  unsigned int* hist;             // sort_hist_len(nblocks) entries
  int nblocks;                    // sort_grid(): blocks that are resident together
  unsigned int* bar;              // barrier arrivals, zero before the launch
  StepCounters* ctr;
  BarrierBound bound;
};
int sort_grid(int num_sms);       // 0: the device cannot say
size_t sort_hist_len(int nblocks);
cudaError_t launch_sort(const SortArgs& a, unsigned long long** keys_out, uint32_t** vals_out,
                        cudaStream_t s);
// dst[i] = src[idx[i]] for i < min(ctr->n_out, cap)
cudaError_t launch_permute(const DevHit* src, const uint32_t* idx, DevHit* dst,
                           const StepCounters* ctr, unsigned long long cap, int num_sms,
                           cudaStream_t s);
cudaError_t launch_filter(const StepParams& p, const unsigned long long* sorted, cudaStream_t s);
// Decides carried windows of pairs without hits.
cudaError_t launch_finalize(const StepParams& p, const unsigned long long* sorted,
                            cudaStream_t s);
// Ordered records (p.ordered).  The scan turns the segment counts into
// offsets (the total into ctr->n_out, overflow bit 2 past cap_out); the emit
// moves the records into dst in canonical order and each work item's first
// record into run_start.  part holds ordered_scan_blocks() entries; p.seg
// must hold ordered_seg_len(p.cap_rtmp) entries, all zero before the filter.
int ordered_scan_blocks(int num_sms);
size_t ordered_seg_len(size_t cap_rtmp);
cudaError_t launch_ordered_scan(const StepParams& p, unsigned long long* part, cudaStream_t s);
cudaError_t launch_ordered_emit(const StepParams& p, const unsigned long long* sorted,
                                DevHit* dst, unsigned long long* run_start, cudaStream_t s);
// The step's new windows and tails into the stream state.
cudaError_t launch_state(const StepParams& p, cudaStream_t s);
// Everything after the candidates of a small step with ordered records, in one
// cooperative launch (p.pair_pool and p.seg need no filling before it).  With
// more than max_cand candidates it ends at once, with more than max_hits hits
// after the verification; *counters then carries kSmallLeft, and the launches
// of other steps go on from there (a thread walks a pair's spanned hits one by
// one while the others wait at a barrier, and that wait is bounded).
struct SmallStep {
  unsigned long long max_cand, max_hits;
  BarrierBound bound;
  DevHit* dst;                    // records in canonical order
  DevHit* direct;                 // pinned host memory for up to direct_cap of them
  unsigned long long direct_cap;  // (more go to dst)
  unsigned long long* run_start;  // pinned host memory, [n_items + 1]
  StepCounters* counters;         // pinned host memory
  unsigned long long* part;       // [nblocks]
  unsigned int* hist;             // sort_hist_len(nblocks)
  unsigned int* bar;              // barrier arrivals, zero before the launch
  unsigned int* sort_bar;
  // set by the launcher
  const unsigned long long* sorted;
  size_t seg_len;
  int lo_bit, hi_bit;
};
int small_step_grid(int num_sms);  // most blocks of the launch; 0: it does not fit
cudaError_t launch_small_step(const StepParams& p, SmallStep a, int nblocks, cudaStream_t s);
// start[w] = first canonically sorted record of work item w, w = 0..n_items
// (start[n_items] = the record count), from the sorted record keys
cudaError_t launch_runs(const unsigned long long* sorted_keys, const StepParams& p,
                        unsigned long long* start, cudaStream_t s);

}  // namespace oasm
